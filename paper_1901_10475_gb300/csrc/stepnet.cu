// stepnet.cu -- a small learned model of each object's time step (not in the
// paper, whose steps adapt inside the serial Alg 3-6; here the step is fixed
// per screen and predicted from the orbital elements).
//
// 8 features -> 64 -> 64 -> 1 (log of the step in seconds), ReLU hidden
// layers, BF16 weights, FP32 accumulation, FP32 master weights updated by
// AdamW.  Parameters, flat FP32: W1[8][64], b1[64], W2[64][64], b2[64],
// w3[64], b3.  Any step keeps the screen sound: every box still bounds its
// whole segment, so the network only trades boxes against candidates.
#include <cuda_bf16.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "scd_internal.cuh"

namespace scd {

constexpr int kIn = SCD_STEPNET_IN, kHid = SCD_STEPNET_HIDDEN;
constexpr int kOffW1 = 0, kOffB1 = kIn * kHid, kOffW2 = kOffB1 + kHid, kOffB2 = kOffW2 + kHid * kHid;
constexpr int kOffW3 = kOffB2 + kHid, kOffB3 = kOffW3 + kHid, kParams = kOffB3 + 1;
static_assert(kParams == SCD_STEPNET_PARAMS, "parameter count");

// ---------------------------------------------------------------------------
// Features of one object, FP32 from the FP64 elements: log(a/R_E), e, sin i,
// cos i, log of perigee and apogee altitude / 100 km, log(P / 1 h), and
// log(1 + number of other objects whose semi-major axis is within 50 km).
// ---------------------------------------------------------------------------
__global__ void k_features(const scd_element *__restrict__ el, int64_t n,
                           const unsigned long long *__restrict__ asorted,
                           float *__restrict__ feat) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  scd_element x = el[i];
  double a = x.a_km, e = x.e;
  double hp = fmax(a * (1.0 - e) - kRe, 1.0), ha = fmax(a * (1.0 + e) - kRe, 1.0);
  double P = kTwoPi * sqrt(a * a * a / kMu);
  // neighbours in semi-major axis: two binary searches in the sorted axes
  double lo_a = a - 50.0, hi_a = a + 50.0;
  int64_t l = 0, h = n;
  while (l < h) {
    int64_t m = (l + h) >> 1;
    if (__longlong_as_double((long long)asorted[m]) < lo_a) l = m + 1; else h = m;
  }
  int64_t first = l;
  l = 0;
  h = n;
  while (l < h) {
    int64_t m = (l + h) >> 1;
    if (__longlong_as_double((long long)asorted[m]) <= hi_a) l = m + 1; else h = m;
  }
  double dens = (double)(l - first - 1);
  float *f = feat + kIn * i;
  f[0] = (float)log(a / kRe);
  f[1] = (float)e;
  f[2] = (float)sin(x.inc_rad);
  f[3] = (float)cos(x.inc_rad);
  f[4] = (float)log(hp / 100.0);
  f[5] = (float)log(ha / 100.0);
  f[6] = (float)log(P / 3600.0);
  f[7] = (float)log1p(fmax(dens, 0.0));
}

__global__ void k_axis_bits(const scd_element *__restrict__ el, int64_t n,
                            unsigned long long *__restrict__ abits) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) abits[i] = (unsigned long long)__double_as_longlong(el[i].a_km);
}

// ---------------------------------------------------------------------------
// Forward pass, one thread per sample; weights in shared memory as BF16.
// ---------------------------------------------------------------------------
struct NetView {
  const __nv_bfloat16 *w1, *w2, *w3;  // BF16 copies
  const float *p;                     // FP32 masters (biases read from here)
};

__global__ void __launch_bounds__(128) k_forward(NetView net, const float *__restrict__ X, int64_t n,
                                                 float *__restrict__ Y) {
  __shared__ __nv_bfloat16 w1[kIn * kHid], w2[kHid * kHid], w3[kHid];
  __shared__ float b1[kHid], b2[kHid];
  for (int k = threadIdx.x; k < kIn * kHid; k += blockDim.x) w1[k] = net.w1[k];
  for (int k = threadIdx.x; k < kHid * kHid; k += blockDim.x) w2[k] = net.w2[k];
  for (int k = threadIdx.x; k < kHid; k += blockDim.x) {
    w3[k] = net.w3[k];
    b1[k] = net.p[kOffB1 + k];
    b2[k] = net.p[kOffB2 + k];
  }
  __syncthreads();
  int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  float x[kIn];
#pragma unroll
  for (int k = 0; k < kIn; ++k) x[k] = X[kIn * s + k];
  float h1[kHid];
#pragma unroll 8
  for (int j = 0; j < kHid; ++j) {
    float acc = b1[j];
#pragma unroll
    for (int k = 0; k < kIn; ++k) acc = fmaf(x[k], __bfloat162float(w1[k * kHid + j]), acc);
    h1[j] = fmaxf(acc, 0.f);
  }
  float y = net.p[kOffB3];
  for (int j = 0; j < kHid; ++j) {
    float acc = b2[j];
#pragma unroll 16
    for (int k = 0; k < kHid; ++k) acc = fmaf(h1[k], __bfloat162float(w2[k * kHid + j]), acc);
    y = fmaf(fmaxf(acc, 0.f), __bfloat162float(w3[j]), y);
  }
  Y[s] = y;
}

// ---------------------------------------------------------------------------
// Forward + backward of the mean squared error over n samples.  A block
// takes tiles of kTS samples; a thread owns two samples by four units of every
// layer (rows ty, ty + 16; see below), so that the three 64 x 64 contractions
// (layer 2, its transpose, its weight gradient) run from registers with one
// 16-byte shared load per four products or better.  The weight gradients stay in
// registers over the block's tiles and leave as one partial per block;
// k_grad sums the partials in a fixed order, so the gradient is the same on
// every run.  Bound by latency (one tile of 32 samples is 0.4 M products, a few
// microseconds): 128 blocks for 4096 samples instead of 32 blocks of
// one-sample threads, two launches and no memsets or copies around them.
// Gradient of 4096 samples through the Python call, loss read back: 155 -> 35
// us.
// ---------------------------------------------------------------------------
constexpr int kTS = 32;       // samples per tile
constexpr int kTT = 256;      // threads: 16 (units) x 16 (samples)
constexpr int kLd = kHid + 4; // padded row of 16-byte words
constexpr int kPart = kParams + 1;  // a block's partial: the gradient, then the loss

struct TrainSmem {
  float W2[kHid][kLd], W1[kIn][kHid];
  float H1[kTS][kLd], D2[kTS][kLd];
  float X[kTS][kIn];
  float w3[kHid], b1[kHid], b2[kHid];
  // block sums of the small gradients: per warp, W1 then b1, b2, w3
  float red[kTT / 32][(kIn + 3) * kHid];
  float tail[kTT / 32][2];  // b3, loss
};

__device__ __forceinline__ float4 ld4(const float *p) {
  return *reinterpret_cast<const float4 *>(p);
}

__global__ void __launch_bounds__(kTT) k_fwd_bwd(NetView net, const float *__restrict__ X,
                                                 const float *__restrict__ T, int64_t n,
                                                 float inv_n, float *__restrict__ part) {
  extern __shared__ __align__(16) unsigned char train_smem[];
  TrainSmem &sm = *reinterpret_cast<TrainSmem *>(train_smem);
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  for (int k = t; k < kHid * kHid; k += kTT)
    sm.W2[k / kHid][k % kHid] = __bfloat162float(net.w2[k]);
  for (int k = t; k < kIn * kHid; k += kTT) (&sm.W1[0][0])[k] = __bfloat162float(net.w1[k]);
  if (t < kHid) {
    sm.w3[t] = __bfloat162float(net.w3[t]);
    sm.b1[t] = net.p[kOffB1 + t];
    sm.b2[t] = net.p[kOffB2 + t];
  }
  const float b3 = net.p[kOffB3];
  // gradients over the block's tiles: W2[4 ty + a][4 tx + b]; W1[.][tx + 16 r],
  // b1[tx + 16 r], b2 and w3[4 tx + b] of the thread's own samples
  float gW2[4][4] = {}, gW1[kIn][4] = {}, gb1[4] = {}, gb2[4] = {}, gw3[4] = {};
  float gb3 = 0.f, loss = 0.f;
  for (int64_t base = (int64_t)blockIdx.x * kTS; base < n; base += (int64_t)gridDim.x * kTS) {
    __syncthreads();  // the weights are in; the tile before is done
    {
      const int64_t q = base * kIn + t;  // kTS * kIn = kTT values
      (&sm.X[0][0])[t] = q < n * kIn ? X[q] : 0.f;
    }
    __syncthreads();
    // layer 1 and 2 of samples ty and ty + 16, units 4 tx .. 4 tx + 3
    {
      float acc[2][4];
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[0][b] = acc[1][b] = sm.b1[4 * tx + b];
#pragma unroll
      for (int k = 0; k < kIn; ++k) {
        const float4 w = ld4(&sm.W1[k][4 * tx]);
        const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[s][b] = fmaf(sm.X[ty + 16 * s][k], wv[b], acc[s][b]);
      }
#pragma unroll
      for (int s = 0; s < 2; ++s)
        *reinterpret_cast<float4 *>(&sm.H1[ty + 16 * s][4 * tx]) =
            make_float4(fmaxf(acc[s][0], 0.f), fmaxf(acc[s][1], 0.f), fmaxf(acc[s][2], 0.f),
                        fmaxf(acc[s][3], 0.f));
    }
    __syncthreads();
    {
      float acc[2][4];
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[0][b] = acc[1][b] = sm.b2[4 * tx + b];
#pragma unroll 4
      for (int k = 0; k < kHid; k += 4) {
        const float4 h0 = ld4(&sm.H1[ty][k]), h1 = ld4(&sm.H1[ty + 16][k]);
        const float hv[2][4] = {{h0.x, h0.y, h0.z, h0.w}, {h1.x, h1.y, h1.z, h1.w}};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float4 w = ld4(&sm.W2[k + c][4 * tx]);
          const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
          for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[s][b] = fmaf(hv[s][c], wv[b], acc[s][b]);
        }
      }
      // the output and its error, per sample over the 16 lanes of its units
      const float4 w3 = ld4(&sm.w3[4 * tx]);
      const float wv[4] = {w3.x, w3.y, w3.z, w3.w};
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        float y = 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          acc[s][b] = fmaxf(acc[s][b], 0.f);
          y = fmaf(acc[s][b], wv[b], y);
        }
#pragma unroll
        for (int d = 8; d > 0; d >>= 1) y += __shfl_xor_sync(0xffffffffu, y, d);
        const int64_t q = base + ty + 16 * s;
        const float r = q < n ? y + b3 - T[q] : 0.f;
        const float dy = 2.f * r * inv_n;
        if (tx == 0) {
          gb3 += dy;
          loss = fmaf(r * inv_n, r, loss);
        }
        float d2[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          gw3[b] = fmaf(dy, acc[s][b], gw3[b]);
          d2[b] = acc[s][b] > 0.f ? dy * wv[b] : 0.f;
          gb2[b] += d2[b];
        }
        *reinterpret_cast<float4 *>(&sm.D2[ty + 16 * s][4 * tx]) =
            make_float4(d2[0], d2[1], d2[2], d2[3]);
      }
    }
    __syncthreads();
    // dW2[k][j] = sum over the samples of h1[k] d2[j]
#pragma unroll 4
    for (int q = 0; q < kTS; ++q) {
      const float4 h = ld4(&sm.H1[q][4 * ty]), d = ld4(&sm.D2[q][4 * tx]);
      const float hv[4] = {h.x, h.y, h.z, h.w}, dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) gW2[a][b] = fmaf(hv[a], dv[b], gW2[a][b]);
    }
    // dL/dpre1 of samples ty, ty + 16, units tx + 16 r (rows of W2 sixteen
    // apart: the 16-byte loads of eight lanes fall into different banks)
    {
      float acc[2][4] = {};
#pragma unroll 4
      for (int j = 0; j < kHid; j += 4) {
        const float4 d0 = ld4(&sm.D2[ty][j]), d1 = ld4(&sm.D2[ty + 16][j]);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float4 w = ld4(&sm.W2[tx + 16 * r][j]);
          acc[0][r] = fmaf(d0.x, w.x, fmaf(d0.y, w.y, fmaf(d0.z, w.z, fmaf(d0.w, w.w, acc[0][r]))));
          acc[1][r] = fmaf(d1.x, w.x, fmaf(d1.y, w.y, fmaf(d1.z, w.z, fmaf(d1.w, w.w, acc[1][r]))));
        }
      }
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float d = sm.H1[ty + 16 * s][tx + 16 * r] > 0.f ? acc[s][r] : 0.f;
          gb1[r] += d;
#pragma unroll
          for (int k = 0; k < kIn; ++k) gW1[k][r] = fmaf(sm.X[ty + 16 * s][k], d, gW1[k][r]);
        }
    }
  }
  // the block's partial: W2 as it stands; the rest summed over the threads
  // of a unit (the warp's two rows by a shuffle, then the eight warps)
  float *out = part + (int64_t)blockIdx.x * kPart;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) out[kOffW2 + (4 * ty + a) * kHid + 4 * tx + b] = gW2[a][b];
  const int w = t >> 5;
  const bool lo = (t & 31) < 16;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
#pragma unroll
    for (int k = 0; k < kIn; ++k) {
      const float v = gW1[k][r] + __shfl_xor_sync(0xffffffffu, gW1[k][r], 16);
      if (lo) sm.red[w][k * kHid + tx + 16 * r] = v;
    }
    const float v1 = gb1[r] + __shfl_xor_sync(0xffffffffu, gb1[r], 16);
    const float v2 = gb2[r] + __shfl_xor_sync(0xffffffffu, gb2[r], 16);
    const float v3 = gw3[r] + __shfl_xor_sync(0xffffffffu, gw3[r], 16);
    if (lo) {
      sm.red[w][kIn * kHid + tx + 16 * r] = v1;
      sm.red[w][(kIn + 1) * kHid + 4 * tx + r] = v2;
      sm.red[w][(kIn + 2) * kHid + 4 * tx + r] = v3;
    }
  }
  gb3 += __shfl_xor_sync(0xffffffffu, gb3, 16);
  loss += __shfl_xor_sync(0xffffffffu, loss, 16);
  if ((t & 31) == 0) {
    sm.tail[w][0] = gb3;
    sm.tail[w][1] = loss;
  }
  __syncthreads();
  for (int e = t; e < (kIn + 3) * kHid + 2; e += kTT) {
    const bool tail = e >= (kIn + 3) * kHid;
    float v = 0.f;
#pragma unroll
    for (int q = 0; q < kTT / 32; ++q)
      v += tail ? sm.tail[q][e - (kIn + 3) * kHid] : sm.red[q][e];
    const int k = e - kIn * kHid;  // b1, b2, w3, then b3 and the loss
    const int at = k < 0          ? kOffW1 + e
                   : k < kHid     ? kOffB1 + k
                   : k < 2 * kHid ? kOffB2 + k - kHid
                                  : kOffW3 + k - 2 * kHid;
    out[at] = v;
  }
}
static_assert(kTS * kIn == kTT && kTS == 32 && kTT == 256, "two samples by four units a thread");
static_assert(kOffB3 == kOffW3 + kHid && kPart == kOffB3 + 2, "b3 and the loss follow w3");

struct AdamArgs {
  float *p, *m, *v;
  int step;
  float lr, wd;
  __nv_bfloat16 *w1, *w2, *w3;
};

// The partials of `blocks` blocks summed in a fixed order, 32 entries by 8
// rows of blocks a thread block; the gradient into g (may be null), the loss
// into host memory the device can write, and with kStep one AdamW step (beta
// 0.9, 0.999, eps 1e-8) on the FP32 masters and the BF16 copies used by the
// forward pass.
constexpr int kGradRows = 8;
template <bool kStep>
__global__ void __launch_bounds__(32 * kGradRows) k_grad(const float *__restrict__ part,
                                                         int blocks, float *__restrict__ g,
                                                         float *loss, AdamArgs a) {
  __shared__ float rows[kGradRows][32];
  const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
  const int k = blockIdx.x * 32 + lane;
  float s = 0.f;
  if (k < kPart)
    for (int b = row; b < blocks; b += kGradRows) s += part[(int64_t)b * kPart + k];
  rows[row][lane] = s;
  __syncthreads();
  if (row > 0 || k >= kPart) return;
  float gk = 0.f;
#pragma unroll
  for (int q = 0; q < kGradRows; ++q) gk += rows[q][lane];
  if (k == kParams) {
    *loss = gk;
    return;
  }
  if (g) g[k] = gk;
  if constexpr (kStep) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float mk = b1 * a.m[k] + (1.f - b1) * gk;
    const float vk = b2 * a.v[k] + (1.f - b2) * gk * gk;
    a.m[k] = mk;
    a.v[k] = vk;
    const float mh = mk / (1.f - powf(b1, (float)a.step));
    const float vh = vk / (1.f - powf(b2, (float)a.step));
    const bool is_weight =
        k < kOffB1 || (k >= kOffW2 && k < kOffB2) || (k >= kOffW3 && k < kOffB3);
    float pk = a.p[k];
    if (is_weight) pk -= a.lr * a.wd * pk;  // decoupled weight decay (weights only)
    pk -= a.lr * mh / (sqrtf(vh) + eps);
    a.p[k] = pk;
    if (k < kOffB1) a.w1[k - kOffW1] = __float2bfloat16_rn(pk);
    else if (k >= kOffW2 && k < kOffB2) a.w2[k - kOffW2] = __float2bfloat16_rn(pk);
    else if (k >= kOffW3 && k < kOffB3) a.w3[k - kOffW3] = __float2bfloat16_rn(pk);
  }
}

__global__ void k_refresh_bf16(const float *__restrict__ p, __nv_bfloat16 *__restrict__ w1,
                               __nv_bfloat16 *__restrict__ w2, __nv_bfloat16 *__restrict__ w3) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < kIn * kHid) w1[k] = __float2bfloat16_rn(p[kOffW1 + k]);
  if (k < kHid * kHid) w2[k] = __float2bfloat16_rn(p[kOffW2 + k]);
  if (k < kHid) w3[k] = __float2bfloat16_rn(p[kOffW3 + k]);
}

// per-object learned step [s]: exp of the network output, clamped to
// [P/400, P/50]
__global__ void k_learned_steps(const scd_element *__restrict__ el, const float *__restrict__ y,
                                int64_t n, float *__restrict__ ks) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double a = el[i].a_km;
  double P = kTwoPi * sqrt(a * a * a / kMu);
  double k = exp((double)y[i]);
  k = fmin(fmax(k, P / 400.0), P / 50.0);
  ks[i] = (float)k;
}

}  // namespace scd

using namespace scd;

struct scd_stepnet {
  cudaStream_t stream = nullptr;
  DevBuf<float> p, m, v, part;
  DevBuf<__nv_bfloat16> w1, w2, w3;
  int step = 0;
  float *h_loss = nullptr;  // pinned: the gradient kernel writes the loss into it
};

static int net_ok(const scd_stepnet *n) { return n && n->p.p; }

static NetView view(const scd_stepnet *n) {
  NetView v;
  v.w1 = n->w1.p;
  v.w2 = n->w2.p;
  v.w3 = n->w3.p;
  v.p = n->p.p;
  return v;
}

static int refresh(scd_stepnet *n) {
  k_refresh_bf16<<<(kHid * kHid + 255) / 256, 256, 0, n->stream>>>(n->p.p, n->w1.p, n->w2.p,
                                                                   n->w3.p);
  note_launch();
  return cudaGetLastError() == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}

extern "C" SCD_API int scd_stepnet_create(void *cuda_stream, uint64_t seed, scd_stepnet **out) {
  if (!out) return SCD_ERR_INVALID_ARG;
  *out = nullptr;
  scd_stepnet *n = new scd_stepnet();
  n->stream = (cudaStream_t)cuda_stream;
  cudaStream_t st = n->stream;
  if (!n->p.ensure(kParams, st) || !n->m.ensure(kParams, st) || !n->v.ensure(kParams, st) ||
      !n->w1.ensure(kIn * kHid, st) ||
      !n->w2.ensure(kHid * kHid, st) || !n->w3.ensure(kHid, st) ||
      cudaMallocHost(&n->h_loss, sizeof(float)) != cudaSuccess) {
    scd_stepnet_destroy(n);
    return SCD_ERR_OOM;
  }
  // He-style initialisation from a host counter-based generator (splitmix64)
  std::vector<float> h(kParams, 0.f);
  uint64_t x = seed;
  auto uni = [&x]() {
    x += 0x9e3779b97f4a7c15ull;
    uint64_t z = x;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    z ^= z >> 31;
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);
  };
  for (int k = 0; k < kIn * kHid; ++k) h[kOffW1 + k] = (float)((2 * uni() - 1) * sqrt(6.0 / kIn));
  for (int k = 0; k < kHid * kHid; ++k) h[kOffW2 + k] = (float)((2 * uni() - 1) * sqrt(6.0 / kHid));
  for (int k = 0; k < kHid; ++k) h[kOffW3 + k] = (float)((2 * uni() - 1) * sqrt(3.0 / kHid));
  int rc = scd_stepnet_set_params(n, h.data(), kParams);
  if (rc) {
    scd_stepnet_destroy(n);
    return rc;
  }
  *out = n;
  return SCD_OK;
}

extern "C" SCD_API int scd_stepnet_set_params(scd_stepnet *n, const float *host_params,
                                              int64_t count) {
  if (!net_ok(n) || !host_params || count != kParams) return SCD_ERR_INVALID_ARG;
  cudaStream_t st = n->stream;
  if (cudaMemcpyAsync(n->p.p, host_params, sizeof(float) * kParams, cudaMemcpyHostToDevice, st) !=
          cudaSuccess ||
      cudaMemsetAsync(n->m.p, 0, sizeof(float) * kParams, st) != cudaSuccess ||
      cudaMemsetAsync(n->v.p, 0, sizeof(float) * kParams, st) != cudaSuccess)
    return SCD_ERR_CUDA;
  n->step = 0;
  int rc = refresh(n);
  if (rc) return rc;
  return cudaStreamSynchronize(st) == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}

extern "C" SCD_API int scd_stepnet_get_params(const scd_stepnet *n, float *host_params,
                                              int64_t count) {
  if (!net_ok(n) || !host_params || count != kParams) return SCD_ERR_INVALID_ARG;
  if (cudaMemcpyAsync(host_params, n->p.p, sizeof(float) * kParams, cudaMemcpyDeviceToHost,
                      n->stream) != cudaSuccess)
    return SCD_ERR_CUDA;
  return cudaStreamSynchronize(n->stream) == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}

extern "C" SCD_API int scd_stepnet_features(const scd_element *d_elems, int64_t n, float *d_feat,
                                            void *cuda_stream) {
  if (!d_elems || n <= 0 || !d_feat) return SCD_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  DevBuf<unsigned long long> ab;
  SortScratch sc;
  if (!ab.ensure(n, st)) return SCD_ERR_OOM;
  k_axis_bits<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(d_elems, n, ab.p);
  note_launch();
  int rc = radix_sort_u64(ab.p, nullptr, n, 64, sc, st);
  if (rc == SCD_OK) {
    k_features<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(d_elems, n, ab.p, d_feat);
    note_launch();
    rc = cudaGetLastError() == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
  }
  cudaStreamSynchronize(st);
  ab.release(st);
  sc.release(st);
  return rc;
}

extern "C" SCD_API int scd_stepnet_forward(const scd_stepnet *n, const float *d_x, int64_t count,
                                           float *d_y) {
  if (!net_ok(n) || !d_x || !d_y || count < 0) return SCD_ERR_INVALID_ARG;
  if (count == 0) return SCD_OK;
  k_forward<<<(unsigned)((count + 127) / 128), 128, 0, n->stream>>>(view(n), d_x, count, d_y);
  note_launch();
  return cudaGetLastError() == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}

// The gradient of the mean squared error into g (may be null) and the loss
// into n->h_loss; with `adam` one optimiser step.
static int train_pass(scd_stepnet *n, const float *d_x, const float *d_t, int64_t count, float *g,
                      const AdamArgs *adam) {
  cudaStream_t st = n->stream;
  static PerDevice waves;
  const int wave = waves.get(
      current_device(), [] { return resident_blocks(k_fwd_bwd, kTT, sizeof(TrainSmem)); });
  const int blocks = (int)std::min<int64_t>((count + kTS - 1) / kTS, wave);
  if (!n->part.ensure((size_t)blocks * kPart, st)) return SCD_ERR_OOM;
  k_fwd_bwd<<<blocks, kTT, sizeof(TrainSmem), st>>>(view(n), d_x, d_t, count,
                                                    1.0f / (float)count, n->part.p);
  const int gb = (kPart + 31) / 32;
  if (adam)
    k_grad<true><<<gb, 32 * kGradRows, 0, st>>>(n->part.p, blocks, g, n->h_loss, *adam);
  else
    k_grad<false><<<gb, 32 * kGradRows, 0, st>>>(n->part.p, blocks, g, n->h_loss, AdamArgs{});
  note_launch(2);
  return cudaGetLastError() == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}

extern "C" SCD_API int scd_stepnet_grad(scd_stepnet *n, const float *d_x, const float *d_t,
                                        int64_t count, float *d_grad, float *loss_out) {
  if (!net_ok(n) || !d_x || !d_t || !d_grad || count <= 0) return SCD_ERR_INVALID_ARG;
  int rc = train_pass(n, d_x, d_t, count, d_grad, nullptr);
  if (rc) return rc;
  if (cudaStreamSynchronize(n->stream) != cudaSuccess) return SCD_ERR_CUDA;
  if (loss_out) *loss_out = *n->h_loss;
  return SCD_OK;
}

extern "C" SCD_API int scd_stepnet_train_step(scd_stepnet *n, const float *d_x, const float *d_t,
                                              int64_t count, float lr, float weight_decay,
                                              float *loss_out) {
  if (!net_ok(n) || !d_x || !d_t || count <= 0 || !(lr > 0.f) || weight_decay < 0.f)
    return SCD_ERR_INVALID_ARG;
  const AdamArgs adam{n->p.p, n->m.p, n->v.p, n->step + 1, lr, weight_decay,
                      n->w1.p, n->w2.p, n->w3.p};
  int rc = train_pass(n, d_x, d_t, count, nullptr, &adam);
  if (rc) return rc;
  n->step += 1;
  if (loss_out) {
    if (cudaStreamSynchronize(n->stream) != cudaSuccess) return SCD_ERR_CUDA;
    *loss_out = *n->h_loss;
  }
  return SCD_OK;
}

// checkpoint: 8-byte magic, version, parameter count, AdamW step, then the
// FP32 master parameters
static const char kMagic[8] = {'S', 'C', 'D', 'N', 'E', 'T', '0', '1'};

extern "C" SCD_API int scd_stepnet_save(const scd_stepnet *n, const char *path) {
  if (!net_ok(n) || !path) return SCD_ERR_INVALID_ARG;
  std::vector<float> h(kParams);
  int rc = scd_stepnet_get_params(n, h.data(), kParams);
  if (rc) return rc;
  FILE *f = fopen(path, "wb");
  if (!f) return SCD_ERR_INVALID_ARG;
  int32_t hdr[3] = {1, kParams, n->step};
  bool ok = fwrite(kMagic, 1, 8, f) == 8 && fwrite(hdr, sizeof(int32_t), 3, f) == 3 &&
            fwrite(h.data(), sizeof(float), kParams, f) == (size_t)kParams;
  ok = (fclose(f) == 0) && ok;
  return ok ? SCD_OK : SCD_ERR_INVALID_ARG;
}

extern "C" SCD_API int scd_stepnet_load(scd_stepnet *n, const char *path) {
  if (!net_ok(n) || !path) return SCD_ERR_INVALID_ARG;
  FILE *f = fopen(path, "rb");
  if (!f) return SCD_ERR_INVALID_ARG;
  char mg[8];
  int32_t hdr[3];
  std::vector<float> h(kParams);
  bool ok = fread(mg, 1, 8, f) == 8 && memcmp(mg, kMagic, 8) == 0 &&
            fread(hdr, sizeof(int32_t), 3, f) == 3 && hdr[0] == 1 && hdr[1] == kParams &&
            fread(h.data(), sizeof(float), kParams, f) == (size_t)kParams;
  fclose(f);
  if (!ok) return SCD_ERR_INVALID_ARG;
  return scd_stepnet_set_params(n, h.data(), kParams);
}

extern "C" SCD_API void scd_stepnet_destroy(scd_stepnet *n) {
  if (!n) return;
  cudaStream_t st = n->stream;
  cudaStreamSynchronize(st);
  n->p.release(st); n->m.release(st); n->v.release(st); n->part.release(st);
  n->w1.release(st); n->w2.release(st); n->w3.release(st);
  if (n->h_loss) cudaFreeHost(n->h_loss);
  delete n;
}

namespace scd {
// learned steps [s] of a scene's objects (LEARNED policy), into s->d_learned
int learned_steps(scd_scene *s) {
  const scd_stepnet *net = (const scd_stepnet *)s->stepnet;
  if (!net_ok(net)) return SCD_ERR_INVALID_ARG;
  cudaStream_t st = s->stream;
  if (!s->d_feat.ensure((size_t)kIn * s->n, st) || !s->d_learned.ensure(s->n, st) ||
      !s->d_ny.ensure(s->n, st))
    return SCD_ERR_OOM;
  int rc = scd_stepnet_features(s->d_el.p, s->n, s->d_feat.p, (void *)st);
  if (rc) return rc;
  // the network runs on the scene's stream
  k_forward<<<(unsigned)((s->n + 127) / 128), 128, 0, st>>>(view(net), s->d_feat.p, s->n,
                                                           s->d_ny.p);
  k_learned_steps<<<(unsigned)((s->n + 255) / 256), 256, 0, st>>>(s->d_el.p, s->d_ny.p, s->n,
                                                                   s->d_learned.p);
  note_launch(2);
  return cudaGetLastError() == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}
}  // namespace scd

namespace scd {
__global__ void k_count_per_object(const scd_pair *__restrict__ pr, int64_t n, int64_t nobj,
                                   uint32_t *__restrict__ cnt) {
  int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  scd_pair q = pr[k];
  if ((int64_t)q.i < nobj) atomicAdd(cnt + q.i, 1u);
  if ((int64_t)q.j < nobj) atomicAdd(cnt + q.j, 1u);
}
}  // namespace scd

extern "C" SCD_API int scd_count_pairs_per_object(const scd_pair *d_pairs, int64_t n_pairs,
                                                  int64_t n_objects, uint32_t *d_counts,
                                                  void *cuda_stream) {
  if (n_pairs < 0 || n_objects <= 0 || !d_counts || (n_pairs > 0 && !d_pairs))
    return SCD_ERR_INVALID_ARG;
  if (n_pairs == 0) return SCD_OK;
  k_count_per_object<<<(unsigned)((n_pairs + 255) / 256), 256, 0, (cudaStream_t)cuda_stream>>>(
      d_pairs, n_pairs, n_objects, d_counts);
  note_launch();
  return cudaGetLastError() == cudaSuccess ? SCD_OK : SCD_ERR_CUDA;
}
