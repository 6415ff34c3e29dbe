// lbvh.cu -- steps A6-A7: the 4D box hierarchy.  The paper's AABB tree
// (Sec. 3.2) is built there by incremental insertion; here the boxes are
// sorted along a 4D Hilbert curve and the tree over them is implicit (every
// eight consecutive nodes of a level under one node of the next, packed as a
// Hilbert R-tree is: Kamel & Faloutsos 1994), so building it is one bottom-up
// reduction: no links, no arrival counts, no search for split points.
#include <algorithm>

#include "scd_internal.cuh"

namespace scd {

// One block takes 512 nodes of level k0 (the sorted boxes when k0 = 0) and
// builds the three levels above them: 64 nodes, 8 nodes, one node.  The
// boxes of the topmost nodes go to the next launch (k0 + 3), 1/512 of the size,
// or, where they fit one tile, to the last block to finish.  Bound
// by the gather's loads: 32 bytes a box read at random (two 16-byte halves, a
// sector each) and 32 + 4 written, 14 bytes of nodes.  With the neighbour
// links 0.69 ms for 17.4 M boxes (a binary radix tree with its gather and
// bottom-up refit took 2.34 ms).
constexpr int kTreeThreads = kWide * kWide * kWide;

struct TreeArgs {
  // level 0: the boxes by id, and what the gather writes of each
  const uint32_t *id;
  const float4 *lo, *hi;
  const uint32_t *obj;
  const unsigned long long *keys;  // sorted keys (cells only)
  int cell_shift;
  SBox *sbox;
  uint32_t *sobj, *posof, *scell;
  // levels above: boxes of level k0 in, of level k0 + 3 out
  const SBox *in;
  SBox *out;
  WideNode *nodes;
  TreeLevels lv;
  int k0;
  int64_t n;                       // boxes (a capacity when d_n is set)
  const unsigned long long *d_n;
  // set: the levels above k0 + 3 fit one tile, and the last block to finish
  // builds them (zero before and after the launch)
  uint32_t *finish;
};

__device__ __forceinline__ float4 f4min(float4 a, float4 b) {
  return make_float4(fminf(a.x, b.x), fminf(a.y, b.y), fminf(a.z, b.z), fminf(a.w, b.w));
}
__device__ __forceinline__ float4 f4max(float4 a, float4 b) {
  return make_float4(fmaxf(a.x, b.x), fmaxf(a.y, b.y), fmaxf(a.z, b.z), fmaxf(a.w, b.w));
}
__device__ __forceinline__ float4 f4_xor_lane(float4 a, int d) {
  return make_float4(__shfl_xor_sync(0xffffffffu, a.x, d), __shfl_xor_sync(0xffffffffu, a.y, d),
                     __shfl_xor_sync(0xffffffffu, a.z, d), __shfl_xor_sync(0xffffffffu, a.w, d));
}

// One axis of a node's frame: its own extent onto cells 1.25 to 126.25 of 127
// (whole cells 1 to 126; 0 and 127 are outside).  Ticks (whole numbers): onto
// the middles of cells, one cell per tick while the node spans at most 125 of
// them, so that consecutive segments, which touch without overlapping, stay
// apart.
__device__ __forceinline__ void axis_frame(float lo, float hi, bool tick, float &scale,
                                           float &off) {
  const float ext = hi - lo;
  scale = tick ? (125.0f / kCellTop) / fmaxf(ext, 125.0f) : (125.0f / kCellTop) / ext;
  off = (tick ? 1.5f : 1.25f) / kCellTop - lo * scale;
  // (an infinite extent would map finite faces to a cell above infinite ones)
  if (!isfinite(ext) || !isfinite(scale) || !isfinite(off)) scale = off = 0.0f;
}

// Eight neighbouring lanes hold a node's children (valid: the child exists);
// the node is put together in shared memory and (lo, hi) become its own box.
// Called by whole warps.
__device__ __forceinline__ void make_node(float4 &lo, float4 &hi, bool valid, WideNode *dst) {
  const float inf = __int_as_float(0x7f800000);
  const int c = threadIdx.x & (kWide - 1);
  const float4 cl = lo, ch = hi;
  if (!valid) {
    lo = make_float4(inf, inf, inf, inf);
    hi = make_float4(-inf, -inf, -inf, -inf);
  }
#pragma unroll
  for (int d = 1; d < kWide; d <<= 1) {
    lo = f4min(lo, f4_xor_lane(lo, d));
    hi = f4max(hi, f4_xor_lane(hi, d));
  }
  float4 s, o;
  axis_frame(lo.x, hi.x, false, s.x, o.x);
  axis_frame(lo.y, hi.y, false, s.y, o.y);
  axis_frame(lo.z, hi.z, false, s.z, o.z);
  axis_frame(lo.w, hi.w, true, s.w, o.w);
  unsigned char *bl = reinterpret_cast<unsigned char *>(dst->half[c >> 2].lo) + (c & 3);
  unsigned char *bh = reinterpret_cast<unsigned char *>(dst->half[c >> 2].hi) + (c & 3);
  // a child that does not exist: lower faces above all, upper ones below
  bl[0] = valid ? (unsigned char)node_coord(cl.x, s.x, o.x, false) : 127;
  bl[4] = valid ? (unsigned char)node_coord(cl.y, s.y, o.y, false) : 127;
  bl[8] = valid ? (unsigned char)node_coord(cl.z, s.z, o.z, false) : 127;
  bl[12] = valid ? (unsigned char)node_coord(cl.w, s.w, o.w, false) : 127;
  bh[0] = valid ? (unsigned char)node_coord(ch.x, s.x, o.x, true) : 128;
  bh[4] = valid ? (unsigned char)node_coord(ch.y, s.y, o.y, true) : 128;
  bh[8] = valid ? (unsigned char)node_coord(ch.z, s.z, o.z, true) : 128;
  bh[12] = valid ? (unsigned char)node_coord(ch.w, s.w, o.w, true) : 128;
  if (c == 0) {
    *reinterpret_cast<float4 *>(dst->scale) = s;
    *reinterpret_cast<float4 *>(dst->off) = o;
  }
}

struct TreeSmem {
  WideNode s1[kWide * kWide], s2[kWide], s3;
  SBox u1[kWide * kWide], u2[kWide];
};

// The three levels above 512 nodes of level k0 (tile of them), whose boxes
// are gathered by id (k0 = 0) or read from `in`; the topmost node's box goes
// to `out`.
template <bool kGather>
__device__ __forceinline__ void tree_tile(const TreeArgs &a, TreeSmem &sm, int k0, int64_t n,
                                          int64_t tile, const SBox *in, SBox *out) {
  // nodes of level k0 and of the two above
  const int s0 = kWideBits * k0;
  const int64_t c0 = (n + (1ll << s0) - 1) >> s0, c1 = (c0 + 7) >> 3, c2 = (c1 + 7) >> 3;
  const int tid = threadIdx.x;
  const int64_t i = tile * kTreeThreads + tid;
  const bool valid = i < c0;
  float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
  if (valid) {
    if (kGather) {
      const uint32_t b = a.id[i];
      lo = __ldg(a.lo + b);
      hi = __ldg(a.hi + b);
      a.sbox[i].lo = lo;
      a.sbox[i].hi = hi;
      if (a.sobj) a.sobj[i] = __ldg(a.obj + b);
      // a box referenced from several cells: any copy will do, their data agree
      if (a.posof) a.posof[b] = (uint32_t)i;
      if (a.scell) a.scell[i] = (uint32_t)(a.keys[i] >> a.cell_shift);
    } else {  // (past L1: other blocks may have written it in this launch)
      lo = __ldcg(&in[i].lo);
      hi = __ldcg(&in[i].hi);
    }
  }
  make_node(lo, hi, valid, &sm.s1[tid >> 3]);
  if ((tid & 7) == 0) {
    sm.u1[tid >> 3].lo = lo;
    sm.u1[tid >> 3].hi = hi;
  }
  __syncthreads();
  // whole nodes out, 16 bytes a thread
  auto store = [&](const WideNode *src, int level, int64_t first, int64_t count) {
    uint4 *dst = reinterpret_cast<uint4 *>(a.nodes + a.lv.off[level] + first);
    const uint4 *from = reinterpret_cast<const uint4 *>(src);
    for (int k = tid; k < (int)count * 6; k += kTreeThreads) dst[k] = from[k];
  };
  store(sm.s1, k0 + 1, tile * 64, c1 - tile * 64 < 64 ? c1 - tile * 64 : 64);
  if (k0 + 2 <= a.lv.levels) {
    if (tid < kWide * kWide) {
      lo = sm.u1[tid].lo;
      hi = sm.u1[tid].hi;
      make_node(lo, hi, tile * 64 + tid < c1, &sm.s2[tid >> 3]);
      if ((tid & 7) == 0) {
        sm.u2[tid >> 3].lo = lo;
        sm.u2[tid >> 3].hi = hi;
      }
    }
    __syncthreads();
    store(sm.s2, k0 + 2, tile * 8, c2 - tile * 8 < 8 ? c2 - tile * 8 : 8);
  }
  if (k0 + 3 <= a.lv.levels) {
    if (tid < 32) {
      // every eight lanes put together the same node
      lo = sm.u2[tid & 7].lo;
      hi = sm.u2[tid & 7].hi;
      make_node(lo, hi, tile * 8 + (tid & 7) < c2, &sm.s3);
      if (tid == 0) {
        out[tile].lo = lo;
        out[tile].hi = hi;
      }
    }
    __syncthreads();
    store(&sm.s3, k0 + 3, tile, 1);
  }
  __syncthreads();  // the next tile reuses the shared nodes
}

// (three blocks an SM: at 58 registers two fit, 0.77 ms instead of 0.69 for the
// tree and the links)
template <bool kGather>
__global__ void __launch_bounds__(kTreeThreads, 3) k_tree(TreeArgs a) {
  __shared__ TreeSmem sm;
  __shared__ bool last;
  int64_t n = a.n;
  if (a.d_n && *a.d_n < (unsigned long long)n) n = (int64_t)*a.d_n;
  const int s3 = kWideBits * (a.k0 + 3);
  const int64_t tiles = (n + (1ll << s3) - 1) >> s3;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x)
    tree_tile<kGather>(a, sm, a.k0, n, tile, a.in, a.out);
  if (!a.finish) return;
  // the last block to get here sees every block's topmost boxes
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(a.finish, 1u) == gridDim.x - 1u;
    if (last) {
      *a.finish = 0u;
      __threadfence();
    }
  }
  __syncthreads();
  if (last && tiles > 0) tree_tile<false>(a, sm, a.k0 + 3, n, 0, a.out, a.out + tiles);
}

// Each sorted box's object and the sorted positions of that object's previous
// and next segments (-1 at the ends of the horizon).  Adjacent segments lie
// close in space and time, so these positions stay near p along the curve.
// (In object order everything read lies in order, but 16 bytes written at
// random cost more than the reads: 0.5 ms against 0.17 for 17.4 M boxes.)
__global__ void k_links(const uint32_t *__restrict__ id, const uint32_t *__restrict__ obj,
                        const uint32_t *__restrict__ posof, int64_t Nq, int64_t nbox,
                        int4 *__restrict__ out) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= Nq) return;
  const int64_t u = (int64_t)id[p];
  const uint32_t o = obj[u];
  const int prev = u > 0 && obj[u - 1] == o ? (int)posof[u - 1] : -1;
  const int next = u + 1 < nbox && obj[u + 1] == o ? (int)posof[u + 1] : -1;
  out[p] = make_int4(prev, next, (int)o, 0);
}

int64_t tree_scratch_boxes(int64_t cap) {
  int64_t total = 0;
  for (int64_t c = (cap + kTreeThreads - 1) / kTreeThreads;; c = (c + kTreeThreads - 1) / kTreeThreads) {
    total += c;
    if (c <= 1) return total;
  }
}

// the launches of one tree: level 0 with the gather, then three levels each
static int launch_tree(TreeArgs a, SBox *nbox, cudaStream_t st) {
  static PerDevice waves;
  const int wave =
      waves.get(current_device(), [] { return resident_blocks(k_tree<true>, kTreeThreads); });
  a.lv = tree_levels(a.n);
  int64_t tiles = (a.n + kTreeThreads - 1) / kTreeThreads;
  uint32_t *const finish = a.finish;
  a.in = nullptr;
  a.out = nbox;
  for (a.k0 = 0; a.k0 < a.lv.levels; a.k0 += 3) {
    // one tile of topmost nodes (up to 2^18 boxes at the first launch, 2^27 at
    // the second): the same launch builds the levels above them
    const bool ends = a.k0 + 3 < a.lv.levels && tiles <= kTreeThreads;
    a.finish = ends ? finish : nullptr;
    // with a device count, one resident wave loops over the tiles there are
    const unsigned grid = (unsigned)(a.d_n ? std::min<int64_t>(tiles, wave) : tiles);
    if (a.k0 == 0) k_tree<true><<<grid, kTreeThreads, 0, st>>>(a);
    else k_tree<false><<<grid, kTreeThreads, 0, st>>>(a);
    note_launch();
    if (ends) break;
    a.in = a.out;
    a.out += tiles;
    tiles = (tiles + kTreeThreads - 1) / kTreeThreads;
  }
  return cudaGetLastError() == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}

int build_tree(scd_scene *s, const unsigned long long *keys_sorted, const uint32_t *ids_sorted,
               int64_t Nq, int cell_shift) {
  cudaStream_t st = s->stream;
  const bool cells = cell_shift >= 0;
  if (!s->s_box.ensure(Nq, st) || !s->d_posof.ensure(s->N, st) || !s->s_link.ensure(Nq, st) ||
      !s->d_nodes.ensure(tree_levels(Nq).total, st) ||
      !s->d_nbox.ensure(tree_scratch_boxes(Nq), st) || (cells && !s->s_cell.ensure(Nq, st)))
    return SCD_ERR_OOM;
  TreeArgs a{};
  a.id = ids_sorted;
  a.lo = s->d_lo.p;
  a.hi = s->d_hi.p;
  a.obj = s->d_obj.p;
  a.keys = keys_sorted;
  a.cell_shift = cells ? cell_shift : 0;
  a.sbox = s->s_box.p;
  a.posof = s->d_posof.p;
  a.scell = cells ? s->s_cell.p : nullptr;
  a.nodes = s->d_nodes.p;
  a.n = Nq;
  a.finish = &s->d_ctr.p->tree_done;
  if (int rc = launch_tree(a, s->d_nbox.p, st)) return rc;
  const int bs = 256;
  k_links<<<(unsigned)((Nq + bs - 1) / bs), bs, 0, st>>>(ids_sorted, s->d_obj.p, s->d_posof.p, Nq,
                                                         s->N, s->s_link.p);
  note_launch();
  return cudaGetLastError() == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}

// One refinement round's sorted boxes and the tree over them: up to cap
// boxes, their count on the device.
int build_round_tree(const uint32_t *ids_sorted, const float4 *lo, const float4 *hi,
                     const uint32_t *obj, int64_t cap, const unsigned long long *d_M, SBox *sbox,
                     uint32_t *sobj, WideNode *nodes, SBox *nbox, DevCounters *ctr,
                     cudaStream_t st) {
  TreeArgs a{};
  a.id = ids_sorted;
  a.lo = lo;
  a.hi = hi;
  a.obj = obj;
  a.sbox = sbox;
  a.sobj = sobj;
  a.nodes = nodes;
  a.n = cap;
  a.d_n = d_M;
  a.finish = &ctr->tree_done;
  return launch_tree(a, nbox, st);
}

int build_hierarchy(scd_scene *s) {
  return build_tree(s, nullptr, s->d_id.p, s->N, -1);
}

}  // namespace scd
