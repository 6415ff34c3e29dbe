// traverse.cu -- step A8: every box queries the hierarchy for the boxes it
// meets (the tree query of Sec. 3.2, run for all boxes at once) and the
// candidate records are emitted; step A9: the canonical list.
//
// Each box pair is found once: box p only visits nodes that hold a later
// sorted position, and of those only later boxes.
//
// Merged output without sorting the raw set: for one object pair the tick
// intersections of their overlapping box pairs ("cells") are disjoint and
// tile the horizon in order, so a merged interval is a maximal run of
// consecutive overlapping cells.  Every hit looks at the cell just before it
// (one segment back on whichever object's segment begins at the cell's first
// tick) and the cell just after it (one segment forward on whichever ends at
// its last tick).  A run's first cell emits a start record; if that cell is
// also the run's last, the record is "closed" and carries the last tick,
// else it is "open" and the run's last cell emits an end record.  After the
// starts and the ends are sorted by (i, j, tick), the k-th open start pairs
// with the k-th end.  The last tick is packed below the start's key when
// 2 (object bits + tick bits) <= 64 and an all-ones tick field cannot be a
// tick (the open tag), else it travels as a 32-bit sort value.
#include <algorithm>
#include <type_traits>

#include "scd_internal.cuh"

namespace scd {

struct TravArgs {
  const WideNode *nodes;      // the tree (all levels, lv.off)
  TreeLevels lv;
  const SBox *sbox;           // sorted boxes
  const uint32_t *sobj, *sid; // (rounds) object and unsorted id of each sorted box
  const int4 *link;           // (screens) previous / next segment (-1: none), object, 0
  int64_t N;
  int T;
  int raw;
  int obj_bits, t_bits;
  int packed;                 // run starts carry their last tick in the low t_bits
  uint32_t open_tag;          // last tick of an open run start
  unsigned long long *starts, *ends;
  uint32_t *rawval;           // raw cells' (or unpacked run starts') last tick
  uint32_t cap;               // record slots (slot_cap)
  uint32_t chunk;             // slots reserved at a time
  DevCounters *ctr;
  // static decomposition (kind SCD_DECOMP_NONE: one tree over all boxes)
  int dkind;
  int n_slabs, p_bands;
  const uint32_t *scell;     // cell of each sorted reference
  const int32_t *cellend;    // one past the last reference of each cell
  const double2 *rr;         // radial ranges (ALT_BANDS)
  const double *edges;       // band edges (ALT_BANDS)
  const int32_t *objT;       // per-object horizon (a batch of scenes), or null
  // refinement rounds (kRefine): the box count on the device (N is the
  // capacity), a flag word per interval (indexed by unsorted id) and the
  // round's candidates (tick candidates, or spans at the finest level of
  // the continuous variant)
  const unsigned long long *d_N;
  uint32_t *rflags;
  unsigned long long *rcand, *rncand;
  unsigned long long rcap;
  int rspans;
};

// Is `cell` the one cell that reports the overlapping pair (q, b)?  The
// lower corner of the boxes' intersection (SLAB_OCT), or the lower end of
// the two objects' common radial range (ALT_BANDS, which also drops pairs
// with no potential-collision edge).
__device__ __forceinline__ bool reports_here(const TravArgs &a, uint32_t cell, float4 ql, float4 bl,
                                             uint32_t qo, uint32_t bo) {
  if (a.dkind == SCD_DECOMP_SLAB_OCT) {
    float cx = fmaxf(ql.x, bl.x), cy = fmaxf(ql.y, bl.y), cz = fmaxf(ql.z, bl.z);
    int64_t ct = (int64_t)fmaxf(ql.w, bl.w);
    uint32_t c = (uint32_t)(slab_of(ct, a.n_slabs, a.T) * 8 + ((cx >= 0.f) << 2) +
                            ((cy >= 0.f) << 1) + (cz >= 0.f));
    return c == cell;
  }
  if (a.dkind == SCD_DECOMP_ALT_BANDS) {
    double2 r1 = a.rr[qo], r2 = a.rr[bo];
    double lo = fmax(r1.x, r2.x), hi = fmin(r1.y, r2.y);
    return lo <= hi && (uint32_t)band_of(lo, a.edges, a.p_bands) == cell;
  }
  return true;
}

// a slot that holds no record: all key bits set, so it sorts after every
// real record (whose object fields can never be all ones)
constexpr unsigned long long kHole = ~0ull;

// Whole-warp emission into a chunk of slots reserved by the warp (one atomic
// per chunk).  A chunk's unused tail is filled with holes, which the record
// sorts carry along, so small screens take small chunks: at most half as
// many slots as boxes a warp (3001 objects, 2 h: 2.5 M slots of 512 for 0.46 M
// records).  Every lane of the warp calls put() together; the chunk state is
// warp-uniform.
constexpr unsigned kMinChunk = 32, kMaxChunk = 512;
struct ChunkCursor {
  uint32_t next, end, count;
};

__device__ __forceinline__ void chunk_fill_holes(ChunkCursor &c, unsigned long long *buf,
                                                 uint32_t cap) {
  const int lane = threadIdx.x & 31;
  for (uint32_t k = c.next + lane; k < c.end; k += 32)
    if (k < cap) buf[k] = kHole;
}

__device__ __forceinline__ void chunk_put(ChunkCursor &c, unsigned long long *buf, uint32_t *vbuf,
                                          unsigned long long *slots, uint32_t cap, uint32_t chunk,
                                          bool pred, unsigned long long key, uint32_t v) {
  const int lane = threadIdx.x & 31;
  const unsigned vote = __ballot_sync(0xffffffffu, pred);
  const uint32_t cnt = __popc(vote);
  if (cnt == 0) return;
  uint32_t next = c.next;
  if (next + cnt > c.end) {
    chunk_fill_holes(c, buf, cap);
    uint32_t b = 0;
    if (lane == 0) b = chunk_first(atomicAdd(slots, (unsigned long long)chunk), chunk);
    next = __shfl_sync(0xffffffffu, b, 0);
    if (lane == 0) c.end = next + chunk;
  }
  if (pred) {
    const uint32_t idx = next + __popc(vote & ((1u << lane) - 1u));
    if (idx < cap) {
      buf[idx] = key;
      if (vbuf) vbuf[idx] = v;
    }
  }
  __syncwarp();
  if (lane == 0) {
    c.next = next + cnt;
    c.count += cnt;
  }
  __syncwarp();
}

// Is (q, b) the first / last cell of its run?  Both need the neighbouring
// cell: one segment back (forward) on whichever box starts (ends) there,
// found by sorted position (close to the pair along the curve, so the loads
// hit cache).
__device__ __forceinline__ void run_ends_sorted(const TravArgs &a, float4 ql0, float4 qh0,
                                                int2 qn, float4 bl, float4 bh, int2 bn, int s,
                                                int e, int T, bool &start, bool &end) {
  int qt0 = (int)ql0.w, qt1 = (int)qh0.w, bt0 = (int)bl.w, bt1 = (int)bh.w;
  if (start && s > 0) {
    float4 ql = ql0, qh = qh0, cl = bl, ch = bh;
    if (qt0 == s) ldg_box(a.sbox + qn.x, ql, qh);
    if (bt0 == s) ldg_box(a.sbox + bn.x, cl, ch);
    start = !box_overlap(ql, qh, cl, ch);
  }
  if (end && e < T) {
    float4 ql = ql0, qh = qh0, cl = bl, ch = bh;
    if (qt1 == e) ldg_box(a.sbox + qn.y, ql, qh);
    if (bt1 == e) ldg_box(a.sbox + bn.y, cl, ch);
    end = !box_overlap(ql, qh, cl, ch);
  }
}

__device__ __forceinline__ unsigned long long pair_key(const TravArgs &a, uint32_t oa,
                                                       uint32_t ob) {
  unsigned long long i = min(oa, ob), j = max(oa, ob);
  return (i << (a.obj_bits + a.t_bits)) | (j << a.t_bits);
}

// A start record: (i, j, first tick), with the run's last tick (or the open
// tag) packed below it; `last` is also the sort value when unpacked.
__device__ __forceinline__ unsigned long long start_key(const TravArgs &a, unsigned long long pk,
                                                        int s, uint32_t last) {
  unsigned long long key = pk | (unsigned long long)s;
  return a.packed ? (key << a.t_bits) | (unsigned long long)last : key;
}

// ---------------------------------------------------------------------------
// Persistent traversal.  Every loop iteration of every lane is the same step
// (load one node, test its eight children), so lanes stay in lock step; a
// lane whose query is done takes the next one from a pool its warp claims in
// blocks; leaf nodes with overlapping boxes go to a per-warp buffer and the
// records of their pairs are worked out by the whole warp together, into
// output chunks the warp reserves.
//
// kGroup neighbouring lanes walk together: their queries are consecutive along
// the curve and visit nearly the same nodes, so the group visits the union of
// them and one load serves its lanes.  A group's pending nodes are one 32-bit
// word per level (the parent's index and a mask of its children still to
// visit; 64 bits above 2^30 boxes): one a level in shared memory, whatever the
// query, so no stack
// can overflow.
//
// Bound by the L1's wavefronts (its data pipe is busy 90% of the time, the
// schedulers 66%): a node's three 32-byte loads take one each per distinct
// line, and so do a pair's exact boxes, links and neighbouring segments.
// 24 h catalog screen (17.4 M boxes, 164 M runs; SPEED / INTERVAL boxes):
// 10.1 / 5.15 ms.  What led here, measured at one stage or another: lanes alone
// 12.2 / 6.5, groups of two 11.3 / 5.9, of four 11.6 / 6.1, of eight 14.1 / 7.7;
// 256 buffered leaf nodes instead of 160, SPEED 11.5 to 11.3; a pair's object
// and links in one load, with the registers it takes, 11.2 / 5.9 to 10.6 /
// 5.3; the pairs left over by one expansion joining the next, 10.4 / 5.26; the
// record chunks' state in shared memory, so that eight blocks of 64 registers
// fit without spills, 10.1 / 5.15.  Slower: fetching the children ahead into
// L1 (17.7 / 15.8), the neighbours' rounded boxes beside the links (12.9 /
// 5.8), two lanes testing half the children each for both (a sixth fewer
// wavefronts, 18% more instructions; 10.4 / 5.36).  Two-child nodes of 36 bytes
// along a Morton curve, with 64-entry stacks in local memory, took 18.4 / 10.7
// and 91 nodes a query.
// ---------------------------------------------------------------------------
constexpr int kTvThreads = 128;
constexpr int kTvWarps = kTvThreads / 32;
// lanes that walk together (their queries are consecutive)
constexpr int kGroup = 2;
// lanes without a query before the warp hands out new ones, a step of the whole
// warp (INTERVAL 5.31 -> 5.25 ms; SPEED the same; 2 and 8 lie between)
constexpr int kMinRefill = 4;
// leaf nodes (query, node, mask of its boxes) buffered per warp, drained when
// fewer than one step's worth (32) of slots remain
constexpr int kEntryCap = 256;
// entries expanded into single pairs at a time, two per lane
constexpr int kExpand = 64;
// queries claimed per warp atomic; small, so that the queries in flight stay
// a narrow window of the curve and their nodes stay in L2
constexpr unsigned kQueryChunk = 32;
// a refill can hand out up to 32 queries at once, from the pool's rest and
// one new chunk: a chunk smaller than a warp would leave lanes without one
static_assert(kQueryChunk >= 32, "a query chunk covers at least one warp's refill");

// (in shared memory: the registers go to the pairs)
struct WarpEmit {
  ChunkCursor s, e;  // start and end record chunks (raw cells use s)
};

// A pair whose boxes meet in a node's frame, decided on the exact boxes.
// Refinement rounds: both intervals of a pair of meeting boxes of different
// objects are flagged; two single ticks that meet (the same tick) are a tick
// candidate, and at the finest level of the continuous variant every meeting
// pair is a span.
__device__ __forceinline__ void round_pair(const TravArgs &a, uint32_t p, uint32_t b) {
  float4 ql, qh, bl, bh;
  ldg_box(a.sbox + p, ql, qh);
  ldg_box(a.sbox + b, bl, bh);
  const uint32_t qo = __ldg(a.sobj + p), bo = __ldg(a.sobj + b);
  if (bo == qo || !box_overlap(ql, qh, bl, bh)) return;
  const bool longq = qh.w > ql.w, longb = bh.w > bl.w;
  atomicOr(a.rflags + __ldg(a.sid + p), kRfHit | (longb ? kRfHitLong : 0u));
  atomicOr(a.rflags + __ldg(a.sid + b), kRfHit | (longq ? kRfHitLong : 0u));
  unsigned long long key;
  if (a.rspans) {
    key = rf_span_key(min(qo, bo), max(qo, bo), (int32_t)ql.w, (int32_t)bl.w);
  } else if (!longq && !longb) {
    key = rf_tick_key((uint32_t)ql.w, min(qo, bo), max(qo, bo));
  } else {
    return;
  }
  const unsigned long long q = atomicAdd(a.rncand, 1ull);
  if (q < a.rcap) a.rcand[q] = key;
}

// The screen's pairs, one per lane (valid: the lane has one); called by the
// whole warp.
__device__ __forceinline__ void screen_pair(const TravArgs &a, bool valid, uint32_t p, uint32_t b,
                                            WarpEmit &we) {
  float4 ql = make_float4(0.f, 0.f, 0.f, 0.f), qh = ql, bl = ql, bh = ql;
  uint32_t qo = 0, bo = 0;
  int4 qk = make_int4(0, 0, 0, 0), bk = qk;
  if (valid) {
    ldg_box(a.sbox + p, ql, qh);
    qk = __ldg(a.link + p);
    ldg_box(a.sbox + b, bl, bh);
    bk = __ldg(a.link + b);
    qo = (uint32_t)qk.z;
    bo = (uint32_t)bk.z;
    valid = bo != qo && box_overlap(ql, qh, bl, bh);
    if (valid && a.dkind != SCD_DECOMP_NONE)
      valid = reports_here(a, __ldg(a.scell + p), ql, bl, qo, bo);
  }
  int s = max((int)ql.w, (int)bl.w), e = min((int)qh.w, (int)bh.w);
  unsigned long long pk = pair_key(a, qo, bo);
  if (a.raw) {
    chunk_put(we.s, a.starts, a.rawval, &a.ctr->n_raw, a.cap, a.chunk, valid,
              pk | (unsigned long long)s, (uint32_t)e);
    return;
  }
  bool start = valid, end = valid;
  if (valid)
    run_ends_sorted(a, ql, qh, make_int2(qk.x, qk.y), bl, bh, make_int2(bk.x, bk.y), s, e,
                    a.objT ? __ldg(a.objT + qo) : a.T, start, end);
  const uint32_t last = end ? (uint32_t)e : a.open_tag;
  chunk_put(we.s, a.starts, a.packed ? nullptr : a.rawval, &a.ctr->n_starts, a.cap,
            a.chunk, start,
            start_key(a, pk, s, last), last);
  chunk_put(we.e, a.ends, nullptr, &a.ctr->n_ends, a.cap, a.chunk, end && !start,
            pk | (unsigned long long)e, 0u);
}

// a warp's buffered leaf nodes and the pairs they are expanded into
struct HitBuf {
  uint32_t p[kEntryCap], n[kEntryCap];  // query, leaf node
  uint8_t mask[kEntryCap];              // its boxes that meet the query
  uint16_t pair[kExpand * kWide + 32];  // entry | box << 8
};
static_assert(kEntryCap <= 256, "an expanded pair names its entry in eight bits");

// The buffered leaf nodes' pairs, spread evenly over the lanes: the entries'
// boxes are counted and listed kExpand entries at a time, then 32 listed
// pairs at a time are decided; fewer than 32 left over go with the next
// entries.  Returns the pairs.
template <bool kRefine>
__device__ __forceinline__ int drain(const TravArgs &a, HitBuf &h, int cnt, WarpEmit &we) {
  const int lane = threadIdx.x & 31;
  int pairs = 0, rest = 0;
  for (int base = 0; base < cnt; base += kExpand) {
    const int k0 = base + lane, k1 = k0 + 32;
    uint32_t m0 = k0 < cnt ? h.mask[k0] : 0u, m1 = k1 < cnt ? h.mask[k1] : 0u;
    // exclusive position of the lane's pairs
    const int mine = __popc(m0) + __popc(m1);
    int at = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, at, d);
      if (lane >= d) at += v;
    }
    const int total = rest + __shfl_sync(0xffffffffu, at, 31);
    at += rest - mine;
    for (; m0; m0 &= m0 - 1u) h.pair[at++] = (uint16_t)(k0 | (__ffs(m0) - 1) << 8);
    for (; m1; m1 &= m1 - 1u) h.pair[at++] = (uint16_t)(k1 | (__ffs(m1) - 1) << 8);
    __syncwarp();
    // whole warps of pairs; the rest goes with the next entries
    const int now = base + kExpand < cnt ? total & ~31 : total;
    for (int r = 0; r < now; r += 32) {
      const bool valid = r + lane < total;
      uint32_t p = 0, b = 0;
      if (valid) {
        const uint32_t code = h.pair[r + lane];
        p = h.p[code & 255u];
        b = h.n[code & 255u] * kWide + (code >> 8);
      }
      if constexpr (kRefine) {
        if (valid) round_pair(a, p, b);
      } else {
        screen_pair(a, valid, p, b, we);
      }
    }
    pairs += now;
    rest = total - now;
    const uint16_t left = lane < rest ? h.pair[now + lane] : (uint16_t)0;
    __syncwarp();
    if (lane < rest) h.pair[lane] = left;
  }
  return pairs;
}

// The children of a node that the query box meets in the node's frame, as a
// mask: 16 FP32 operations bring the query's faces into the frame, then per
// axis and four children one byte-wise difference each tests lo <= query hi
// and query lo <= hi (the guard bit survives where it holds).
__device__ __forceinline__ uint32_t meet_mask(const WideNode *nd, float4 qlo, float4 qhi) {
  uint32_t f[8], c0[8], c1[8];
  ldg_words(nd->scale, f);
  ldg_words(&nd->half[0], c0);
  ldg_words(&nd->half[1], c1);
  const float ql[4] = {qlo.x, qlo.y, qlo.z, qlo.w}, qh[4] = {qhi.x, qhi.y, qhi.z, qhi.w};
  uint32_t r0 = 0x80808080u, r1 = 0x80808080u;
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    const float sc = __uint_as_float(f[d]), of = __uint_as_float(f[4 + d]);
    const uint32_t l4 = __byte_perm(node_coord(ql[d], sc, of, false), 0u, 0x0000u);
    const uint32_t h4 = __byte_perm(node_coord(qh[d], sc, of, true), 0u, 0x0000u);
    r0 &= (h4 - c0[d]) & (c0[4 + d] - l4);
    r1 &= (h4 - c1[d]) & (c1[4 + d] - l4);
  }
  // the guard bits of children 0-3 and 4-7 gathered into the top byte: bit
  // 8 c and bit 8 c + 4 of x go to 24 + c and 28 + c (no two products of the
  // multiplication share a bit)
  const uint32_t x = ((r0 >> 7) & 0x01010101u) | ((r1 >> 3) & 0x10101010u);
  return (x * 0x01020408u) >> 24;
}

template <bool kRefine, bool kHuge>
__global__ void __launch_bounds__(kTvThreads, 8) k_traverse(TravArgs a) {
  __shared__ HitBuf hits[kTvWarps];
  using Word = typename std::conditional<kHuge, unsigned long long, uint32_t>::type;
  constexpr int kLevels = kHuge ? kMaxLevels : kWordLevels;
  __shared__ Word pend[kLevels][kTvThreads / kGroup];  // [level - 1]: parent << 8 | mask
  __shared__ uint32_t off[kMaxLevels + 1];
  constexpr unsigned kFull = 0xffffffffu;
  constexpr int kStride = kTvThreads / kGroup;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int sub = lane & (kGroup - 1);
  const unsigned lt = (1u << lane) - 1u;
  constexpr unsigned kLead = 0x55555555u;  // the groups' first lanes
  static_assert(kGroup == 2, "kLead and the group reduction are for pairs of lanes");
  HitBuf &buf = hits[w];
  Word *const mine = &pend[0][threadIdx.x / kGroup] - kStride;  // level l at mine[l * kStride]
  if (threadIdx.x <= kMaxLevels) off[threadIdx.x] = a.lv.off[threadIdx.x];
  __syncthreads();
  int nent = 0;  // warp-uniform
  uint32_t visits = 0;
  uint32_t ntests = 0;
  uint32_t p = 0;     // current query (sorted position)
  uint32_t cend = 0;  // one past the last position it may meet (0: no query)
  uint32_t lv = 0;    // the group's levels with pending nodes; 0 = no query
  float4 qlo = make_float4(0.f, 0.f, 0.f, 0.f), qhi = qlo;
  bool dry = false;   // warp-uniform: the queue is empty
  // the last box has no later partner: queries are 0 .. N-2
  const int64_t nbox = kRefine && a.d_N && *a.d_N < (unsigned long long)a.N ? (int64_t)*a.d_N
                                                                            : a.N;
  const uint32_t nq = nbox > 1 ? (uint32_t)(nbox - 1) : 0u;
  // the warp's query pool: the first chunk by the warp's place in the grid,
  // the later ones by the counter (no atomics where a few warps do it all)
  uint32_t q_next = min((blockIdx.x * kTvWarps + w) * kQueryChunk, nq);
  uint32_t q_end = q_next + kQueryChunk;
  __shared__ WarpEmit emits[kTvWarps];
  WarpEmit &we = emits[w];
  if (lane == 0) we.s = we.e = ChunkCursor{0, 0, 0};
  __syncwarp();
  for (;;) {
    unsigned idle = __ballot_sync(kFull, lv == 0u);
    if (idle && (dry || __popc(idle) >= kMinRefill)) {
      if (!dry) {
        // groups without queries take the next ones from the warp's pool
        const uint32_t cnt = (uint32_t)__popc(idle);  // whole groups are idle
        const uint32_t have = q_end - q_next;
        uint32_t nb = 0;
        if (have < cnt) {
          const unsigned long long later = (unsigned long long)gridDim.x * kTvWarps * kQueryChunk;
          unsigned long long c = 0;
          if (later < (unsigned long long)nq) {
            if (lane == 0) c = atomicAdd(&a.ctr->work_next, (unsigned long long)kQueryChunk);
            c = __shfl_sync(kFull, c, 0);
          }
          c += later;
          dry = c >= (unsigned long long)nq;
          nb = dry ? nq : (uint32_t)c;
        }
        const uint32_t r = (uint32_t)__popc(idle & lt);
        const uint32_t q = r < have ? q_next + r : nb + (r - have);
        uint32_t gend = 0;
        if (lv == 0u) {
          cend = 0;
          if (q < nq) {
            p = q;
            ldg_box(a.sbox + p, qlo, qhi);
            cend = (uint32_t)nbox;
            if (!kRefine && a.dkind != SCD_DECOMP_NONE)
              cend = (uint32_t)__ldg(a.cellend + __ldg(a.scell + p));
            if (p + 1u >= cend) cend = 0;  // the last of its cell
          }
          gend = cend;
        }
        // the group's end (its queries may lie in several cells) and start
        gend = max(gend, __shfl_xor_sync(kFull, gend, 1));
        const uint32_t p0 = q - (uint32_t)sub;
        if (lv == 0u && gend > 0u) {
          // start at the smallest node that holds p0 and the last position
          const int h = (kWideBits + 31 - __clz((int)(p0 ^ (gend - 1u)))) / kWideBits;
          const uint32_t top = kHuge ? (uint32_t)((unsigned long long)p0 >> (kWideBits * h))
                                     : p0 >> (kWideBits * h);
          mine[h * kStride] = (Word)(top >> kWideBits) << 8 | 1u << (top & 7u);
          lv = 1u << h;
        }
        if (have < cnt) {
          q_next = nb + (cnt - have);
          q_end = nb + kQueryChunk;
        } else {
          q_next += cnt;
        }
        __syncwarp();
      } else {
        // The queue is empty: an idle group takes pending nodes of a group
        // that has some to spare, with its queries: the whole word of its
        // highest level, or the last child of its only one; long queries then
        // spread over the warp instead of holding it.
        if (idle == kFull) break;
        const int hl = lv ? 31 - __clz((int)lv) : 0;
        const Word word = lv ? mine[hl * kStride] : 0u;
        const bool more = (lv & (lv - 1u)) != 0u;  // a lower level has some too
        idle &= kLead;
        const unsigned donors =
            __ballot_sync(kFull, more || __popc((uint32_t)word & 0xffu) > 1) & kLead;
        const int moves = min(__popc(idle), __popc(donors));
        if (moves > 0) {
          const int lead = lane - sub;  // the group's first lane
          const unsigned lb = (1u << lead) - 1u;
          const int ri = __popc(idle & lb), rd = __popc(donors & lb);
          const bool take = ((idle >> lead) & 1u) && ri < moves;
          const bool give = ((donors >> lead) & 1u) && rd < moves;
          const uint32_t top = 0x80u >> (__clz((int)((uint32_t)word & 0xffu)) - 24);  // last child's bit
          const Word part = more ? word : (word & ~(Word)0xffu) | top;
          // the receiver of rank k takes from the donor of rank k
          int src = lane;
          if (take) {
            unsigned m = donors;
            for (int k = 0; k < ri; ++k) m &= m - 1u;
            src = __ffs(m) - 1 + sub;
          }
          const Word gword = __shfl_sync(kFull, part, src);
          const int glevel = __shfl_sync(kFull, hl, src);
          p = __shfl_sync(kFull, p, src);
          cend = __shfl_sync(kFull, cend, src);
          qlo.x = __shfl_sync(kFull, qlo.x, src);
          qlo.y = __shfl_sync(kFull, qlo.y, src);
          qlo.z = __shfl_sync(kFull, qlo.z, src);
          qlo.w = __shfl_sync(kFull, qlo.w, src);
          qhi.x = __shfl_sync(kFull, qhi.x, src);
          qhi.y = __shfl_sync(kFull, qhi.y, src);
          qhi.z = __shfl_sync(kFull, qhi.z, src);
          qhi.w = __shfl_sync(kFull, qhi.w, src);
          if (give) {
            if (more) lv ^= 1u << hl;
            else mine[hl * kStride] = word ^ top;
          }
          if (take) {
            mine[glevel * kStride] = gword;
            lv = 1u << glevel;
          }
          __syncwarp();
        }
      }
    }
    // the next pending node of the lowest level
    const bool on = lv != 0u;
    const int l = on ? __ffs(lv) - 1 : 1;
    const Word word = mine[l * kStride];
    __syncwarp();  // read by the whole group before any lane rewrites it
    uint32_t mask = 0, node = 0;
    if (on) {
      const Word rest = word & (word - 1u);
      node = (uint32_t)(word >> 8) * kWide + (__ffs((int)(uint32_t)word) - 1);
      mine[l * kStride] = rest;
      if (!(rest & 0xffu)) lv &= lv - 1u;
      mask = meet_mask(a.nodes + off[l] + node, qlo, qhi);
      ++visits;
      // only children that hold a position in (p, cend)
      const int sh = kWideBits * (l - 1);
      const int lo = (int)((p + 1u) >> sh) - (int)(node * kWide);
      const int hi = (int)((cend - 1u) >> sh) - (int)(node * kWide);
      mask &= (0xffu << min(max(lo, 0), 8)) & ((1u << min(max(hi + 1, 0), 8)) - 1u);
      if (cend == 0u) mask = 0u;
    }
    // the children that a query of the group meets
    const uint32_t any = mask | __shfl_xor_sync(kFull, mask, 1);
    if (on && l > 1 && any) {
      mine[(l - 1) * kStride] = (Word)node << 8 | any;
      lv |= 1u << (l - 1);
    }
    __syncwarp();
    // leaf nodes with boxes that meet go to the warp's buffer
    const bool put = on && l == 1 && mask;
    const unsigned v = __ballot_sync(kFull, put);
    if (v) {
      if (put) {
        const int k = nent + __popc(v & lt);
        buf.p[k] = p;
        buf.n[k] = node;
        buf.mask[k] = (uint8_t)mask;
      }
      nent += __popc(v);
      if (nent > kEntryCap - 32) {
        __syncwarp();
        ntests += drain<kRefine>(a, buf, nent, we);  // exact box tests
        nent = 0;
        // (read again rather than kept in registers across the drain)
        ldg_box(a.sbox + p, qlo, qhi);
      }
    }
  }
  __syncwarp();
  if (nent > 0) ntests += drain<kRefine>(a, buf, nent, we);
  if constexpr (!kRefine) {
    chunk_fill_holes(we.s, a.starts, a.cap);
    if (!a.raw) chunk_fill_holes(we.e, a.ends, a.cap);
  }
  // the block's totals, one atomic each where there is something to add
  unsigned long long nt = (unsigned long long)visits * kWide;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) nt += __shfl_down_sync(0xffffffffu, nt, o);
  __shared__ unsigned long long sums[kTvWarps][4];
  if (lane == 0) {
    sums[w][0] = nt;
    sums[w][1] = ntests;
    sums[w][2] = we.s.count;
    sums[w][3] = we.e.count;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    unsigned long long v = 0;
#pragma unroll
    for (int q = 0; q < kTvWarps; ++q) v += sums[q][threadIdx.x];
    unsigned long long *to = threadIdx.x == 0   ? &a.ctr->node_tests
                             : threadIdx.x == 1 ? &a.ctr->leaf_tests
                             : threadIdx.x == 3 ? &a.ctr->v_ends
                             : a.raw            ? &a.ctr->v_raw
                                                : &a.ctr->v_starts;
    if (v) atomicAdd(to, v);
  }
}

// persistent: as many blocks as fit on the GPU at once
template <bool kRefine, bool kHuge = false>
static int launch_traverse(TravArgs &a, cudaStream_t st) {
  static PerDevice waves;
  const int wave = waves.get(
      current_device(), [] { return resident_blocks(k_traverse<kRefine, kHuge>, kTvThreads); });
  // sorted boxes and nodes are read with 32-byte loads
  if ((reinterpret_cast<uintptr_t>(a.sbox) | reinterpret_cast<uintptr_t>(a.nodes)) & 31)
    return SCD_ERR_INTERNAL;
  a.chunk = kMinChunk;
  while (a.chunk < kMaxChunk && 2 * (int64_t)a.chunk * wave * kTvWarps < a.N) a.chunk *= 2;
  k_traverse<kRefine, kHuge><<<(unsigned)wave, kTvThreads, 0, st>>>(a);
  note_launch();
  return cudaGetLastError() == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}

// One refinement round's traversal over up to cap sorted boxes (their count
// on the device).
int traverse_round(const WideNode *nodes, const SBox *sbox, const uint32_t *sobj,
                   const uint32_t *sid, int64_t cap, const unsigned long long *d_N, int64_t T,
                   DevCounters *ctr, uint32_t *rflags, unsigned long long *rcand,
                   unsigned long long *rncand, unsigned long long rcap, int spans,
                   cudaStream_t st) {
  if (cap < 2) return SCD_OK;
  TravArgs a{};
  a.nodes = nodes;
  a.lv = tree_levels(cap);
  a.sbox = sbox;
  a.sobj = sobj;
  a.sid = sid;
  a.N = cap;
  a.T = (int)T;
  a.ctr = ctr;
  a.dkind = SCD_DECOMP_NONE;
  a.d_N = d_N;
  a.rflags = rflags;
  a.rcand = rcand;
  a.rncand = rncand;
  a.rcap = rcap;
  a.rspans = spans;
  return launch_traverse<true>(a, st);
}

int traverse(scd_scene *s, int raw_mode, int obj_bits, int t_bits) {
  TravArgs a{};
  a.nodes = s->d_nodes.p;
  a.sbox = s->s_box.p;
  a.link = s->s_link.p;
  // one query per sorted reference
  a.N = s->dkind != SCD_DECOMP_NONE ? s->n_refs : s->N;
  a.lv = tree_levels(a.N);
  a.T = (int)s->T;
  a.raw = raw_mode;
  a.obj_bits = obj_bits;
  a.t_bits = t_bits;
  a.packed = !raw_mode && runs_packed(obj_bits, t_bits, s->T);
  a.open_tag = open_tag(a.packed, t_bits);
  a.starts = s->d_starts.p;
  a.ends = s->d_ends.p;
  a.rawval = s->d_rawval.p;
  a.cap = slot_cap(s->pair_cap);
  a.ctr = s->d_ctr.p;
  a.dkind = s->dkind;
  a.n_slabs = s->n_slabs;
  a.p_bands = s->p_bands;
  a.scell = s->s_cell.p;
  a.cellend = s->d_cellend.p;
  a.rr = s->d_rr.p;
  a.edges = s->d_edges.p;
  a.objT = s->n_scenes > 0 ? s->d_objT.p : nullptr;
  return a.lv.levels > kWordLevels ? launch_traverse<false, true>(a, s->stream)
                                   : launch_traverse<false>(a, s->stream);
}

// ---------------------------------------------------------------------------
// Step A9: sort the run starts (or the raw cells) and the run ends by
// (i, j, tick), then unpack the starts; the k-th open start takes the k-th
// end.  Holes sort last, so the first n sorted slots are the n records.
// ---------------------------------------------------------------------------
constexpr int kUpThreads = 256, kUpItems = 8, kUpTile = kUpThreads * kUpItems;

struct UnpackArgs {
  const unsigned long long *starts;  // sorted starts (or raw cells)
  const uint32_t *lastv;             // their last ticks when not packed
  const unsigned long long *ends;    // sorted ends of the open runs
  int64_t n;                         // starts to unpack (a capacity when d_n is set)
  const unsigned long long *d_n;     // the count, when known on the device only
  unsigned long long n_ends;         // ends (a capacity when d_ne is set)
  const unsigned long long *d_ne;
  // the slots handed out for starts and ends, when known on the device only
  const unsigned long long *d_sslots, *d_eslots;
  int ob, tb;
  int packed, raw;
  int w;                             // lowest tick bits the sorts left out
  uint32_t open_tag;
  int64_t tiles;                     // of the capacity
  uint32_t *bcnt;                    // per tile: open starts, then their exclusive prefix
  const uint32_t *open_total;
  scd_pair *out;
  DevCounters *ctr;
};

__device__ __forceinline__ int64_t unpack_count(const UnpackArgs &a) {
  return a.d_n && *a.d_n < (unsigned long long)a.n ? (int64_t)*a.d_n : a.n;
}

// Counts from the device (a replayed find) may have outgrown the capacities they
// were captured for: records are missing then, and holes stand among the first n.
// Nothing is emitted; the host sees the same counts and runs the find again.
__device__ __forceinline__ bool outgrown(const UnpackArgs &a) {
  return a.d_n && (*a.d_sslots > (unsigned long long)a.n || *a.d_eslots > a.n_ends);
}

__device__ __forceinline__ uint32_t last_of(const UnpackArgs &a, unsigned long long key,
                                            int64_t r) {
  return a.packed ? (uint32_t)(key & ((1ull << a.tb) - 1ull)) : __ldg(a.lastv + r);
}

// Tile items are warp-striped: item k of thread t is tile item k * 256 + t,
// so every load and store of a warp is contiguous.

// open starts per tile
__global__ void __launch_bounds__(kUpThreads) k_open_count(UnpackArgs a) {
  if (outgrown(a)) return;  // (the prefix over the tiles is not read either)
  const int64_t n = unpack_count(a);
  __shared__ uint32_t ws[kUpThreads / 32];
  // (past a device count: zeros, which the prefix over all tiles reads)
  for (int64_t tile = blockIdx.x; tile < a.tiles; tile += gridDim.x) {
    const int64_t base = tile * kUpTile + threadIdx.x;
    if (tile * kUpTile >= n) {
      if (threadIdx.x == 0) a.bcnt[tile] = 0;
      continue;
    }
    uint32_t c = 0;
#pragma unroll
    for (int k = 0; k < kUpItems; ++k) {
      int64_t r = base + (int64_t)k * kUpThreads;
      if (r < n) c += last_of(a, __ldg(a.starts + r), r) == a.open_tag;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t t = 0;
      for (int q = 0; q < kUpThreads / 32; ++q) t += ws[q];
      a.bcnt[tile] = t;
    }
    __syncthreads();
  }
}

static_assert(kUpItems * (kUpThreads / 32) == 64, "the tile prefix takes two counts per lane");

// The r-th end in sorted order: the ends stand in the order of (i, j, tick >>
// w), so it is the (r - g0)-th smallest of its group of equal prefixes, which
// starts at g0 (nearly always the end alone).  Ends are distinct, so a group has
// at most 2^w; holes or a longer group are no end (kHole, which no start zips
// with), found within 2^w loads.
__device__ __forceinline__ unsigned long long end_at(const UnpackArgs &a, unsigned long long r,
                                                     unsigned long long n_ends) {
  const unsigned long long e = __ldg(a.ends + r);
  if (a.w == 0 || e == kHole) return e;
  const unsigned long long pre = e >> a.w, most = 1ull << a.w;
  unsigned long long g0 = r, g1 = r + 1;
  while (g0 > 0 && g1 - g0 <= most && (__ldg(a.ends + g0 - 1) >> a.w) == pre) --g0;
  while (g1 < n_ends && g1 - g0 <= most && (__ldg(a.ends + g1) >> a.w) == pre) ++g1;
  if (g1 - g0 == 1) return e;
  if (g1 - g0 > most) return kHole;
  for (unsigned long long x = g0; x < g1; ++x) {
    const unsigned long long v = __ldg(a.ends + x);
    unsigned long long less = 0;
    for (unsigned long long y = g0; y < g1; ++y) less += __ldg(a.ends + y) < v;
    if (less == r - g0) return v;
  }
  return kHole;  // ends that are not distinct
}

// The starts, sorted by all but the lowest w bits of their tick, as pairs in
// the full order.  A group of equal prefixes (the runs of one pair within 2^w
// ticks, at most 2^w of them; mostly 1 to 3) is ranked by counting: each
// start's place is its group's first slot plus the smaller starts in it, and
// an open start's rank among the opens is that of the group's first slot plus
// the smaller opens in it.  A tile's keys lie in shared memory with the 2^w
// before and after it, so that every group is whole; the open runs' ends are
// looked up afterwards, by the whole block.  Bound by instruction issue (70%),
// at twice its bytes' time (8 read and 16 written a pair): 24 h catalog, 164 M
// pairs, 1.69 ms (4.1 GB of DRAM traffic); 55 M pairs 0.45 (0.69 with the ends
// looked up in line and the groups found by comparing neighbours).  A separate
// pass over the keys that sorted the groups in place and a plain unpack took
// 2.05 ms for the 164 M.
constexpr int kUpHalo = 256;  // 2^w at most

__global__ void __launch_bounds__(kUpThreads) k_emit(UnpackArgs a) {
  constexpr int kWarps = kUpThreads / 32;
  __shared__ unsigned long long ks[kUpTile + 2 * kUpHalo];
  __shared__ uint32_t pre[kUpItems * kWarps];   // opens before each warp's 32 slots of the tile
  __shared__ uint32_t mask[kUpItems * kWarps];  // their open starts
  // slots of the same group as the one before them; a word of none on either
  // side of the tile's
  __shared__ uint32_t same[kUpItems * kWarps + 2];
  __shared__ uint2 opens[kUpTile];  // open starts: slot | place + halo << 16, rank among the opens
  __shared__ int nopen;
  if (outgrown(a)) return;
  const int64_t n = unpack_count(a);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned long long tmask = (1ull << a.tb) - 1ull, omask = (1ull << a.ob) - 1ull;
  const unsigned long long n_ends = a.d_ne && *a.d_ne < a.n_ends ? *a.d_ne : a.n_ends;
  if (threadIdx.x == 0) same[0] = same[kUpItems * kWarps + 1] = 0u;
  const int halo = a.w ? 1 << a.w : 0;
  // keys that differ below this bit only are of one group
  const unsigned long long group_size = 1ull << ((a.packed ? a.tb : 0) + a.w);
  if (!a.raw && blockIdx.x == 0 && threadIdx.x == 0 && n > 0 && *a.open_total != n_ends)
    atomicOr(&a.ctr->trav_flags, ERR_ZIP);
  bool bad = false;
  for (int64_t tile = blockIdx.x; tile * kUpTile < n; tile += gridDim.x) {
    const int64_t base = tile * kUpTile;
    if (threadIdx.x == 0) nopen = 0;
    for (int k = threadIdx.x; k < kUpTile + 2 * halo; k += kUpThreads) {
      const int64_t r = base - halo + k;
      if (r >= 0 && r < n) ks[k] = __ldg(a.starts + r);
    }
    __syncthreads();
    // slot x of the tile is ks[halo + x]; slots [first, last) are loaded
    const int first = base >= halo ? -halo : -(int)base;
    const int last = n - base < kUpTile + halo ? (int)(n - base) : kUpTile + halo;
    uint32_t lastv[kUpItems];
#pragma unroll
    for (int k = 0; k < kUpItems; ++k) {
      const int x = k * kUpThreads + threadIdx.x;
      const bool in = x < last;
      lastv[k] = in ? (a.packed ? (uint32_t)(ks[halo + x] & tmask) : __ldg(a.lastv + base + x)) : 0u;
      const unsigned open = __ballot_sync(0xffffffffu, !a.raw && in && lastv[k] == a.open_tag);
      const unsigned join = __ballot_sync(
          0xffffffffu,
          a.w && in && x > first && (ks[halo + x] ^ ks[halo + x - 1]) < group_size);
      if (lane == 0) {
        mask[k * kWarps + w] = open;
        pre[k * kWarps + w] = __popc(open);
        same[k * kWarps + w + 1] = join;
      }
    }
    __syncthreads();
    if (w == 0) {
      // 64 counts, two per lane, scanned in slot order
      const uint32_t c0 = pre[2 * lane], c1 = pre[2 * lane + 1];
      uint32_t x = c0 + c1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      const uint32_t b = (a.raw ? 0u : a.bcnt[tile]) + x - c0 - c1;
      pre[2 * lane] = b;
      pre[2 * lane + 1] = b + c0;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kUpItems; ++k) {
      const int x = k * kUpThreads + threadIdx.x;
      const bool in = x < last;
      const unsigned long long key = in ? ks[halo + x] : 0ull;
      const bool open = (mask[k * kWarps + w] >> lane) & 1u;
      // the group's first slot, its starts below this one, the open ones of
      // them, and the opens of the group before the tile
      int g0 = x, less = 0, oless = 0, obefore = 0;
      if (a.w && in) {
        // the slots of the group around x, from the bits of its 64 neighbours
        const int wd = (x >> 5) + 1, b = x & 31;
        const unsigned long long dn = (unsigned long long)same[wd] << 32 | same[wd - 1];
        const unsigned long long up = (unsigned long long)same[wd + 1] << 32 | same[wd];
        const int below = __clzll(~(dn << (31 - b))), above = __ffsll(~(up >> b >> 1)) - 1;
        g0 = x - below;
        int g1 = x + above + 1;
        if (below > 31 || above > 31 || g0 <= 0 || g1 >= kUpTile) {
          // longer, or at the tile's edge: along the keys
          // (2^w either way at most: more would not be records)
          const int from = max(first, x - halo), to = min(last, x + 1 + halo);
          for (g0 = x; g0 > from && (ks[halo + g0 - 1] ^ key) < group_size;) --g0;
          for (g1 = x + 1; g1 < to && (ks[halo + g1] ^ key) < group_size;) ++g1;
        }
        if (g1 - g0 > 1)
          for (int y = g0; y < g1; ++y) {
            const unsigned long long v = ks[halo + y];
            const int o = (v & tmask) == tmask;
            less += v < key;
            oless += v < key ? o : 0;
            obefore += y < 0 ? o : 0;
          }
      }
      const unsigned long long kk = a.packed ? key >> a.tb : key;
      scd_pair p;
      p.i = (uint32_t)(kk >> (a.ob + a.tb));
      p.j = (uint32_t)((kk >> a.tb) & omask);
      p.tlo = (int32_t)(kk & tmask);
      p.thi = (int32_t)lastv[k];
      // an open run's end is looked up below, by the block together
      const unsigned ov = mask[k * kWarps + w];
      if (ov) {
        int at = 0;
        if (lane == 0) at = atomicAdd(&nopen, __popc(ov));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(ov & ((1u << lane) - 1u));
        if (open) {
          // opens before the group's first slot, in the tile's prefix
          const uint32_t o0 =
              g0 >= 0 ? pre[g0 >> 5] + __popc(mask[g0 >> 5] & ((1u << (g0 & 31)) - 1u))
                      : pre[0] - (uint32_t)obefore;
          opens[at] = make_uint2((uint32_t)x | (uint32_t)(g0 + less + halo) << 16, o0 + oless);
        }
      }
      if (in && !open) a.out[base + g0 + less] = p;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < nopen; q += kUpThreads) {
      const uint2 o = opens[q];
      const unsigned long long key = ks[halo + (o.x & 0xffffu)];
      const unsigned long long kk = a.packed ? key >> a.tb : key;
      scd_pair p;
      p.i = (uint32_t)(kk >> (a.ob + a.tb));
      p.j = (uint32_t)((kk >> a.tb) & omask);
      p.tlo = (int32_t)(kk & tmask);
      p.thi = 0;
      if (o.y < n_ends) {
        const unsigned long long ek = end_at(a, o.y, n_ends);
        p.thi = (int32_t)(ek & tmask);
        bad |= (ek >> a.tb) != (kk >> a.tb) || p.thi <= p.tlo;
      } else {
        bad = true;
      }
      a.out[base - halo + (int)(o.x >> 16)] = p;
    }
    __syncthreads();  // the next tile reuses the keys
  }
  if (bad) atomicOr(&a.ctr->trav_flags, ERR_ZIP);
}

static UnpackArgs unpack_args(scd_scene *s, int raw_mode, int obj_bits, int t_bits) {
  UnpackArgs a{};
  a.starts = s->d_starts.p;
  a.lastv = s->d_rawval.p;
  a.ends = s->d_ends.p;
  a.d_n = nullptr;
  a.d_ne = nullptr;
  a.ob = obj_bits;
  a.tb = t_bits;
  a.raw = raw_mode;
  a.packed = !raw_mode && runs_packed(obj_bits, t_bits, s->T);
  a.open_tag = open_tag(a.packed, t_bits);
  a.out = s->d_out.p;
  a.ctr = s->d_ctr.p;
  return a;
}

static PairEmit pair_emit(scd_scene *s, int obj_bits, int t_bits, const unsigned long long *ends,
                          unsigned long long n_ends, scd_pair *out, int64_t n) {
  PairEmit pe;
  pe.ob = obj_bits;
  pe.tb = t_bits;
  pe.ends = ends;
  pe.n_ends = n_ends;
  pe.out = out;
  pe.n = n;
  pe.flags = &s->d_ctr.p->trav_flags;
  return pe;
}

// k_open_count, the prefix over the tiles, k_emit
static int unpack(scd_scene *s, UnpackArgs a, cudaStream_t st) {
  a.tiles = (a.n + kUpTile - 1) / kUpTile;
  if (a.tiles == 0) return SCD_OK;
  // a block a tile, or with a device count as many as the SMs hold
  const unsigned grid =
      (unsigned)(a.d_n ? std::min<int64_t>(a.tiles, 8 * device_sms()) : a.tiles);
  if (!a.raw) {
    if (!s->d_tilecnt.ensure((size_t)a.tiles + 1, st)) return SCD_ERR_OOM;
    a.bcnt = s->d_tilecnt.p;
    a.open_total = s->d_tilecnt.p + a.tiles;
    k_open_count<<<grid, kUpThreads, 0, st>>>(a);
    scan_u32_exclusive(a.bcnt, a.tiles, s->d_tilecnt.p + a.tiles, st);
    note_launch(2);
  }
  k_emit<<<grid, kUpThreads, 0, st>>>(a);
  note_launch();
  return SCD_OK;
}

// The record sorts skip the lowest w bits of the tick field when that
// saves a whole 8-bit pass (w = the bits of the last, partial digit).  The
// sort is stable, so the records then stand in the order of (i, j, tick >>
// w), each group of equal prefixes in emission order; k_emit ranks each group
// by the whole key.  Records are unique (a pair's runs do not overlap) and
// holes are all ones, so the result is the full sort's order.
static int window_bits(int bits, int t_bits) {
  const int passes = (bits + 7) / 8;
  const int w = bits - 8 * (passes - 1);
  return passes >= 2 && w <= t_bits ? w : 0;
}

int canonicalize(scd_scene *s, int raw_mode, int obj_bits, int t_bits) {
  cudaStream_t st = s->stream;
  // slots to sort (records plus holes) and records to keep
  int64_t ns = raw_mode ? (int64_t)s->h_ctr.n_raw : (int64_t)s->h_ctr.n_starts;
  int64_t n = raw_mode ? (int64_t)s->h_ctr.v_raw : (int64_t)s->h_ctr.v_starts;
  UnpackArgs a = unpack_args(s, raw_mode, obj_bits, t_bits);
  const int lo = a.packed ? t_bits : 0, bits = 2 * obj_bits + t_bits;
  if (!s->d_out.ensure(n > 0 ? n : 1, st)) return SCD_ERR_OOM;
  a.out = s->d_out.p;
  // packed starts and the ends: one pass fewer, the rest in k_emit
  a.w = a.packed && !raw_mode ? window_bits(bits, t_bits) : 0;
  SortOut so;
  int rc = radix_sort_u64(s->d_starts.p, a.packed ? nullptr : s->d_rawval.p, ns, lo + a.w,
                          bits + lo, s->sort_sc, st, &so);
  if (rc) return rc;
  a.starts = (const unsigned long long *)so.keys;
  a.lastv = so.vals;
  if (!raw_mode && s->h_ctr.v_ends > 0) {
    rc = radix_sort_u64(s->d_ends.p, nullptr, (int64_t)s->h_ctr.n_ends, a.w, bits, s->ends_sc, st,
                        &so);
    if (rc) return rc;
    a.ends = (const unsigned long long *)so.keys;
  }
  a.n = n;
  a.n_ends = raw_mode ? 0 : s->h_ctr.v_ends;
  if (int rc2 = unpack(s, a, st)) return rc2;
  s->n_out = n;
  return cudaGetLastError() == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}

// The canonical list for a host destination, in buckets of the pair's
// first object that go to the host while the next ones are sorted: one
// stable pass over the top digit of the starts' and the ends' keys (the top
// bits of i) splits both into digit ranges (starting 16-byte aligned); runs
// of whole digits with about equal numbers of starts form the buckets, and
// each bucket is sorted by the whole key, unpacked into its place in the
// output and copied out on a second stream (the bucket's last sort pass
// writes the pairs themselves: no unpack pass per bucket; for the whole
// list on the device the separate unpack measured faster).  A pair's starts and ends share
// their i, so each bucket zips its own open starts with its own ends.  The
// output equals canonicalize's; one more pass over the records, hidden
// under the copies.
#define TRY_(x)                   \
  do {                            \
    int rc_ = (x);                \
    if (rc_ != SCD_OK) return rc_; \
  } while (0)

int canonicalize_streamed(scd_scene *s, int obj_bits, int t_bits, scd_pair *host) {
  cudaStream_t st = s->stream;
  UnpackArgs a = unpack_args(s, 0, obj_bits, t_bits);
  const int lo = t_bits, bits = 2 * obj_bits + t_bits;
  // the top digit must lie inside the (i, j) fields, so that a pair's open
  // start and its end (different ticks) fall into the same bucket
  if (!a.packed || 2 * obj_bits < 8) return SCD_ERR_STATE;
  const int64_t ns = (int64_t)s->h_ctr.n_starts, n = (int64_t)s->h_ctr.v_starts;
  const int64_t nes = (int64_t)s->h_ctr.n_ends, ne = (int64_t)s->h_ctr.v_ends;
  if (!s->d_out.ensure(n > 0 ? n : 1, st) || !s->d_part.ensure(ns + 256, st) ||
      !s->d_parte.ensure(nes + 256, st))
    return SCD_ERR_OOM;
  if (!s->cstream) {
    if (cudaStreamCreateWithFlags(&s->cstream, cudaStreamNonBlocking) != cudaSuccess)
      return SCD_ERR_CUDA;
    for (int b = 0; b < kStreamBuckets; ++b)
      if (cudaEventCreateWithFlags(&s->cev[b], cudaEventDisableTiming) != cudaSuccess)
        return SCD_ERR_CUDA;
  }
  uint32_t ts[256], te[256];
  TRY_(radix_partition_u64(s->d_starts.p, s->d_part.p, ns, lo + bits - 8, s->sort_sc, ts, st));
  TRY_(radix_partition_u64(s->d_ends.p, s->d_parte.p, nes, bits - 8, s->sort_sc, te, st));
  // digit d's range starts at ps[d] (pe[d]); its records: the keys of the
  // digit, except that the all-ones digit also holds the holes
  int64_t ps[257], pe[257], vs[256], ve[256], sum_s = 0, sum_e = 0;
  ps[0] = pe[0] = 0;
  for (int d = 0; d < 256; ++d) {
    ps[d + 1] = ps[d] + ((ts[d] + 1) & ~1u);
    pe[d + 1] = pe[d] + ((te[d] + 1) & ~1u);
    vs[d] = d < 255 ? ts[d] : n - sum_s;
    ve[d] = d < 255 ? te[d] : ne - sum_e;
    sum_s += vs[d];
    sum_e += ve[d];
  }
  if (vs[255] < 0 || ve[255] < 0 || sum_s != n || sum_e != ne) return SCD_ERR_INTERNAL;
  int64_t out_at = 0;
  int d0 = 0;
  const int nb = stream_buckets(n);
  for (int b = 0; b < nb && d0 < 256; ++b) {
    // whole digits up to about an equal share of the starts still left; the
    // first bucket small, so that the copies (the slower stream) start early
    const int64_t share = b == 0 ? (n + 4 * nb - 1) / (4 * nb)
                                 : (n - out_at + (nb - b) - 1) / (nb - b);
    int d1 = d0;
    int64_t m = 0, me = 0;
    while (d1 < 256 && (m < share || b == nb - 1)) {
      m += vs[d1];
      me += ve[d1];
      ++d1;
    }
    const int64_t slots = ps[d1] - ps[d0], eslots = pe[d1] - pe[d0];
    unsigned long long *ks = s->d_part.p + ps[d0], *ke = s->d_parte.p + pe[d0];
    if (m > 0) {
      if (me > 0) TRY_(radix_sort_u64(ke, nullptr, eslots, bits, s->sort_sc, st));
      TRY_(radix_sort_u64_pairs(ks, slots, lo, bits + lo, s->sort_sc,
                                pair_emit(s, obj_bits, t_bits, ke, (unsigned long long)me,
                                          s->d_out.p + out_at, m),
                                st));
    } else if (me > 0) {
      return SCD_ERR_INTERNAL;  // ends without starts
    }
    if (m > 0) {
      if (cudaEventRecord(s->cev[b], st) != cudaSuccess ||
          cudaStreamWaitEvent(s->cstream, s->cev[b], 0) != cudaSuccess ||
          cudaMemcpyAsync(host + out_at, s->d_out.p + out_at, sizeof(scd_pair) * (size_t)m,
                          cudaMemcpyDeviceToHost, s->cstream) != cudaSuccess)
        return SCD_ERR_CUDA;
    }
    out_at += m;
    d0 = d1;
  }
  if (out_at != n) return SCD_ERR_INTERNAL;
  s->n_out = n;
  return cudaGetLastError() == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}
#undef TRY_

int canonicalize_dev(scd_scene *s, int obj_bits, int t_bits) {
  cudaStream_t st = s->stream;
  const int64_t cap = s->pair_cap;
  if (!s->d_out.ensure(cap, st)) return SCD_ERR_OOM;
  UnpackArgs a = unpack_args(s, 0, obj_bits, t_bits);
  const int lo = a.packed ? t_bits : 0, bits = 2 * obj_bits + t_bits;
  DevCounters *c = s->d_ctr.p;
  a.w = a.packed ? window_bits(bits, t_bits) : 0;
  SortOut so;
  int rc = radix_sort_u64_dev(s->d_starts.p, a.packed ? nullptr : s->d_rawval.p, cap,
                              &c->n_starts, lo + a.w, bits + lo, s->sort_sc, st, &so);
  if (rc) return rc;
  a.starts = (const unsigned long long *)so.keys;
  a.lastv = so.vals;
  rc = radix_sort_u64_dev(s->d_ends.p, nullptr, cap, &c->n_ends, a.w, bits, s->ends_sc, st, &so);
  if (rc) return rc;
  a.ends = (const unsigned long long *)so.keys;
  a.n = cap;
  a.d_n = &c->v_starts;
  a.n_ends = (unsigned long long)cap;
  a.d_ne = &c->v_ends;
  a.d_sslots = &c->n_starts;
  a.d_eslots = &c->n_ends;
  if (int rc2 = unpack(s, a, st)) return rc2;
  return cudaGetLastError() == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}

}  // namespace scd
