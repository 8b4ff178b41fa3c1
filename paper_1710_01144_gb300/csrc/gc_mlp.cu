// Kernels and C ABI of the candidate-proposal network (gc_mlp.cuh):
// features, forward, gradient, Adam, and a minibatch training loop -- all
// float32 kernels on CUDA cores (the tensor cores hold no float32 product, and
// the proposal's training is specified in float32).
#include <limits.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "gc_device.cuh"
#include "gc_internal.cuh"
#include "gc_mlp.cuh"

struct gc_mlp {
  int32_t max_batch = 0;
  cudaStream_t stream = nullptr;
  int slots = 0;                     // CTAs of the tile kernels that are resident at once
  float *params = nullptr;           // [kMlpParams]
  float *grad = nullptr;             // [kMlpGradLen]: the gradient, then the loss
  float *adam_m = nullptr, *adam_v = nullptr;
  float *part = nullptr;             // [min(slots, tiles of max_batch)][kMlpGradLen]
  float *h_grad = nullptr;           // pinned copy of grad
  int64_t t = 0;                     // Adam step count
};

namespace gc {

constexpr int kMlpThreads = 256;

// features of list[i] (i < *m_dev or m) into X[i][8]
__global__ void k_features(const int32_t *__restrict__ list, int32_t m, const int32_t *m_dev,
                           const int32_t *__restrict__ rp, const int32_t *__restrict__ dS,
                           const long long *__restrict__ ub, const int32_t *__restrict__ stamp,
                           const long long *__restrict__ two_hop, const int32_t *__restrict__ mx, int32_t round,
                           long long prev_gain, float *X) {
  const int cnt = m_dev ? *m_dev : m;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += gridDim.x * blockDim.x) {
    float f[kMlpIn];
    cand_features(list[i], rp, dS, ub, stamp, two_hop, mx, round, prev_gain, f);
#pragma unroll
    for (int j = 0; j < kMlpIn; ++j) X[(size_t)i * kMlpIn + j] = f[j];
  }
}

// Scores of few rows: a warp per row, the weights in shared memory.
__global__ void __launch_bounds__(kMlpThreads) k_mlp_forward(const float *__restrict__ W,
                                                             const float *__restrict__ X, int32_t m,
                                                             float *__restrict__ out) {
  __shared__ float sw[kMlpParams];
  __shared__ float sh[kMlpThreads / 32][kMlpHidden];
  for (int i = threadIdx.x; i < kMlpParams; i += blockDim.x) sw[i] = W[i];
  cta_sync();
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gw = blockIdx.x * (blockDim.x >> 5) + wid, nw = gridDim.x * (blockDim.x >> 5);
  for (int s = gw; s < m; s += nw) {
    float x[kMlpIn];
#pragma unroll
    for (int f = 0; f < kMlpIn; ++f) x[f] = X[(size_t)s * kMlpIn + f];
    const float o = mlp_forward_warp(sw, x, sh[wid]);
    if (lane == 0) out[s] = o;
  }
}

// Many rows, and every gradient: rows are taken in tiles of 16 R by CTAs of 256 threads; thread (ty, tx) of
// 16 x 16 computes R rows ty + 16 q by 4 columns of each of the three 64-wide
// products, all of them between shared-memory tiles: activations never reach
// global memory.  GRAD: the CTA keeps its sums of the weight gradients in
// registers over all its tiles (16 of W2, 2 of W1 and one of the 193 others a
// thread) and writes them once, as one row of `part`, which k_mlp_reduce adds.
//
// What bounds it: float32 FMAs against shared-memory loads (6 16-byte loads a
// warp for 32 R FMAs), 28 kFLOP a row, and at small m the latency of one tile.
// So for gradients the small tile is taken while all of them are resident at once
// and the large one, with 2.4 times fewer loads an FMA, beyond; scores alone keep a
// warp per row as long (6 us for 1,024 rows, 9 with tiles; 19 against 12.5 for
// 16,384).  Every sum over inputs or columns runs in the order of one sample by one
// warp (mlp_forward_warp); the sums over rows are per tile and then over tiles.
//
// One warp per row for the activations, stored to memory, and one thread per
// parameter over all rows took 81 us for a gradient of 1,024 rows and 780 us for
// 16,384 on the host's clock; this takes 33 and 56.
constexpr int kMlpPad = kMlpHidden + 4;         // row stride in shared memory: no two rows of a warp share banks
constexpr int kMlpGradLen = kMlpParams + 7;     // a gradient, then its loss (double, 8-byte aligned)
constexpr int kMlpLossAt = kMlpParams + 1;
static_assert(kMlpLossAt % 2 == 0 && kMlpLossAt + 2 <= kMlpGradLen && kMlpGradLen % 2 == 0, "loss alignment");
constexpr int kMlpCtasPerSm = 2;

constexpr size_t mlp_smem(int R) {
  return sizeof(float) * ((size_t)kMlpHidden * kMlpPad + kMlpIn * kMlpHidden + 4 * kMlpHidden +
                          (size_t)16 * R * (4 * kMlpPad + kMlpIn + 2));
}

template <int R, bool GRAD>
__global__ void __launch_bounds__(kMlpThreads, kMlpCtasPerSm)
    k_mlp_tile(const float *__restrict__ W, const float *__restrict__ X, const float *__restrict__ y, int32_t m,
               float *__restrict__ out, float *__restrict__ part) {
  constexpr int T = 16 * R;
  extern __shared__ __align__(16) float smem[];
  float *w2 = smem, *w1 = w2 + kMlpHidden * kMlpPad, *b1 = w1 + kMlpIn * kMlpHidden, *b2 = b1 + kMlpHidden,
        *w3 = b2 + kMlpHidden, *h1 = w3 + 2 * kMlpHidden, *h2 = h1 + T * kMlpPad, *d2 = h2 + T * kMlpPad,
        *d1 = d2 + T * kMlpPad, *x = d1 + T * kMlpPad, *dout = x + T * kMlpIn;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, wid = tid >> 5, lane = tid & 31;
  for (int i = tid; i < kMlpHidden * kMlpHidden; i += kMlpThreads)
    w2[(i / kMlpHidden) * kMlpPad + i % kMlpHidden] = W[kOffW2 + i];
  for (int i = tid; i < kMlpIn * kMlpHidden; i += kMlpThreads) w1[i] = W[kOffW1 + i];
  if (tid < kMlpHidden) {
    b1[tid] = W[kOffB1 + tid];
    b2[tid] = W[kOffB2 + tid];
    w3[tid] = W[kOffW3 + tid];
  }
  const float b3 = W[kOffB3];
  float gw2[4][4] = {}, gw1[2] = {}, gb = 0.f;
  double lsum = 0;
  const int32_t tiles = (int32_t)(((int64_t)m + T - 1) / T);
  for (int32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t r0 = (int64_t)tile * T;
    const int cnt = (int)min((int64_t)T, (int64_t)m - r0);
    cta_sync();  // weights; the last tile's readers
    for (int i = tid; i < T * kMlpIn; i += kMlpThreads) x[i] = i < cnt * kMlpIn ? X[r0 * kMlpIn + i] : 0.f;
    cta_sync();
    {  // h1 = relu(x W1 + b1)
      const float4 b = *(const float4 *)(b1 + 4 * tx);
      float z[R][4];
#pragma unroll
      for (int q = 0; q < R; ++q) z[q][0] = b.x, z[q][1] = b.y, z[q][2] = b.z, z[q][3] = b.w;
#pragma unroll
      for (int f = 0; f < kMlpIn; ++f) {
        const float4 w = *(const float4 *)(w1 + f * kMlpHidden + 4 * tx);
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const float a = x[(ty + 16 * q) * kMlpIn + f];
          z[q][0] = fmaf(a, w.x, z[q][0]);
          z[q][1] = fmaf(a, w.y, z[q][1]);
          z[q][2] = fmaf(a, w.z, z[q][2]);
          z[q][3] = fmaf(a, w.w, z[q][3]);
        }
      }
#pragma unroll
      for (int q = 0; q < R; ++q)
        *(float4 *)(h1 + (ty + 16 * q) * kMlpPad + 4 * tx) =
            make_float4(fmaxf(z[q][0], 0.f), fmaxf(z[q][1], 0.f), fmaxf(z[q][2], 0.f), fmaxf(z[q][3], 0.f));
    }
    cta_sync();
    {  // h2 = relu(h1 W2 + b2)
      const float4 b = *(const float4 *)(b2 + 4 * tx);
      float z[R][4];
#pragma unroll
      for (int q = 0; q < R; ++q) z[q][0] = b.x, z[q][1] = b.y, z[q][2] = b.z, z[q][3] = b.w;
#pragma unroll 4
      for (int k = 0; k < kMlpHidden; k += 4) {
        float4 w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) w[e] = *(const float4 *)(w2 + (k + e) * kMlpPad + 4 * tx);
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const float4 a = *(const float4 *)(h1 + (ty + 16 * q) * kMlpPad + k);
          const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            z[q][0] = fmaf(av[e], w[e].x, z[q][0]);
            z[q][1] = fmaf(av[e], w[e].y, z[q][1]);
            z[q][2] = fmaf(av[e], w[e].z, z[q][2]);
            z[q][3] = fmaf(av[e], w[e].w, z[q][3]);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < R; ++q)
        *(float4 *)(h2 + (ty + 16 * q) * kMlpPad + 4 * tx) =
            make_float4(fmaxf(z[q][0], 0.f), fmaxf(z[q][1], 0.f), fmaxf(z[q][2], 0.f), fmaxf(z[q][3], 0.f));
    }
    cta_sync();
    // out = h2 . W3 + b3, one warp a row
    for (int r = wid; r < cnt; r += kMlpThreads / 32) {
      float o = h2[r * kMlpPad + lane] * w3[lane] + h2[r * kMlpPad + lane + 32] * w3[lane + 32];
#pragma unroll
      for (int q = 16; q > 0; q >>= 1) o += __shfl_xor_sync(0xffffffffu, o, q);
      o += b3;
      if constexpr (!GRAD) {
        if (lane == 0) out[r0 + r] = o;
      } else {
        const float diff = o - y[r0 + r];
        if (lane == 0) {
          dout[r] = 2.f * diff / (float)m;
          lsum += (double)diff * (double)diff;
        }
      }
    }
    if constexpr (GRAD) {
      cta_sync();
      // dL/dz2
      for (int i = tid; i < cnt * kMlpHidden; i += kMlpThreads) {
        const int r = i / kMlpHidden, j = i % kMlpHidden;
        d2[r * kMlpPad + j] = h2[r * kMlpPad + j] > 0.f ? dout[r] * w3[j] : 0.f;
      }
      cta_sync();
      {  // dL/dz1 = (dL/dz2 W2^T) where h1 > 0; columns tx + 16 e: rows of W2 of different banks
        float z[R][4] = {};
#pragma unroll 4
        for (int k = 0; k < kMlpHidden; k += 4) {
          float4 w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) w[e] = *(const float4 *)(w2 + (tx + 16 * e) * kMlpPad + k);
#pragma unroll
          for (int q = 0; q < R; ++q) {
            const float4 a = *(const float4 *)(d2 + (ty + 16 * q) * kMlpPad + k);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              z[q][e] = fmaf(a.x, w[e].x, z[q][e]);
              z[q][e] = fmaf(a.y, w[e].y, z[q][e]);
              z[q][e] = fmaf(a.z, w[e].z, z[q][e]);
              z[q][e] = fmaf(a.w, w[e].w, z[q][e]);
            }
          }
        }
#pragma unroll
        for (int q = 0; q < R; ++q)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int at = (ty + 16 * q) * kMlpPad + tx + 16 * e;
            d1[at] = h1[at] > 0.f ? z[q][e] : 0.f;
          }
      }
      cta_sync();
      // the tile's rows into the gradient; rows past cnt are never read
      float t2[4][4] = {}, t1[2] = {}, tb = 0.f;
#pragma unroll 2
      for (int r = 0; r < cnt; ++r) {
        const float4 a = *(const float4 *)(h1 + r * kMlpPad + 4 * ty), d = *(const float4 *)(d2 + r * kMlpPad + 4 * tx);
        const float av[4] = {a.x, a.y, a.z, a.w}, dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) t2[i][j] = fmaf(av[i], dv[j], t2[i][j]);
        const float xf = x[r * kMlpIn + wid];
        t1[0] = fmaf(xf, d1[r * kMlpPad + lane], t1[0]);
        t1[1] = fmaf(xf, d1[r * kMlpPad + lane + 32], t1[1]);
        if (tid < kMlpHidden) tb += d1[r * kMlpPad + tid];
        else if (tid < 2 * kMlpHidden) tb += d2[r * kMlpPad + tid - kMlpHidden];
        else if (tid < 3 * kMlpHidden) tb = fmaf(h2[r * kMlpPad + tid - 2 * kMlpHidden], dout[r], tb);
        else if (tid == 3 * kMlpHidden) tb += dout[r];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) gw2[i][j] += t2[i][j];
      gw1[0] += t1[0];
      gw1[1] += t1[1];
      gb += tb;
    }
  }
  if constexpr (GRAD) {
    float *p = part + (size_t)blockIdx.x * kMlpGradLen;
    p[kOffW1 + wid * kMlpHidden + lane] = gw1[0];
    p[kOffW1 + wid * kMlpHidden + lane + 32] = gw1[1];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) p[kOffW2 + (4 * ty + i) * kMlpHidden + 4 * tx + j] = gw2[i][j];
    if (tid < kMlpHidden) p[kOffB1 + tid] = gb;
    else if (tid < 2 * kMlpHidden) p[kOffB2 + tid - kMlpHidden] = gb;
    else if (tid < 3 * kMlpHidden) p[kOffW3 + tid - 2 * kMlpHidden] = gb;
    else if (tid == 3 * kMlpHidden) p[kOffB3] = gb;
    __shared__ double sl[kMlpThreads / 32];
    if (lane == 0) sl[wid] = lsum;
    cta_sync();
    if (tid == 0) {
      double t = 0;
      for (int w = 0; w < kMlpThreads / 32; ++w) t += sl[w];
      *(double *)(p + kMlpLossAt) = t;
    }
  }
}

// grad[p] = sum of the rows of part, 32 parameters a CTA (a 128-byte line of
// each row) by 8 groups of rows; the last CTA adds the losses too.  ADAM: the
// step is taken in the same kernel.
template <bool ADAM>
__global__ void __launch_bounds__(kMlpThreads)
    k_mlp_reduce(const float *__restrict__ part, int rows, int32_t m, float *__restrict__ grad, float *p, float *am,
                 float *av, float lr, float b1, float b2, float eps, float c1, float c2) {
  __shared__ float sg[kMlpThreads / 32][32];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, i = blockIdx.x * 32 + lane;
  float acc = 0.f;
  if (i < kMlpParams) {
#pragma unroll 4
    for (int r = wid; r < rows; r += kMlpThreads / 32) acc += part[(size_t)r * kMlpGradLen + i];
  }
  sg[wid][lane] = acc;
  cta_sync();
  if (wid == 0 && i < kMlpParams) {
    float g = 0.f;
#pragma unroll
    for (int w = 0; w < kMlpThreads / 32; ++w) g += sg[w][lane];
    grad[i] = g;
    if constexpr (ADAM) {
      const float mi = b1 * am[i] + (1.f - b1) * g;
      const float vi = b2 * av[i] + (1.f - b2) * g * g;
      am[i] = mi;
      av[i] = vi;
      p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
  }
  if (blockIdx.x == gridDim.x - 1 && wid == 1) {
    double t = 0;
    for (int r = lane; r < rows; r += 32) t += *(const double *)(part + (size_t)r * kMlpGradLen + kMlpLossAt);
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) t += __shfl_xor_sync(0xffffffffu, t, q);
    if (lane == 0) *(double *)(grad + kMlpLossAt) = t / (double)m;
  }
}

// Rows from which tiles of 64 take over.
static bool mlp_large(const gc_mlp *h, int32_t m) { return m > (int64_t)16 * h->slots; }

// Training data for the proposal: the features each evaluated candidate had
// when it was selected (before its bound is replaced) and log1p of the exact
// gain the pruned BFS found.  Appended at *count, up to cap rows.
__global__ void k_record(const int32_t *__restrict__ list, const int32_t *n_sel, const long long *__restrict__ lgain,
                         const int32_t *__restrict__ rp, const int32_t *__restrict__ dS,
                         const long long *__restrict__ ub, const int32_t *__restrict__ stamp,
                         const long long *__restrict__ two_hop, const int32_t *__restrict__ mx, int32_t round,
                         long long prev_gain, float *X, float *y, int32_t cap, int32_t *count) {
  const int m = *n_sel;
  const int base = *(volatile int32_t *)count;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const int row = base + i;
    if (row >= cap) break;
    float f[kMlpIn];
    cand_features(list[i], rp, dS, ub, stamp, two_hop, mx, round, prev_gain, f);
#pragma unroll
    for (int j = 0; j < kMlpIn; ++j) X[(size_t)row * kMlpIn + j] = f[j];
    y[row] = log1pf((float)lgain[i]);
  }
}

__global__ void k_record_advance(const int32_t *n_sel, int32_t cap, int32_t *count) {
  const int c = *count + *n_sel;
  *count = c < cap ? c : cap;
}

int launch_record(gc_graph *g, int32_t round, long long prev_gain) {
  if (!g->rec_X || g->rec_cap <= 0) return GC_OK;
  g->launches += 2;
  k_record<<<g->red_blocks, kRedThreads, 0, g->stream>>>(g->list, &g->sctl->n_sel, g->lgain, g->rp, g->dS, g->ub,
                                                         g->stamp, g->two_hop, g->mx, round, prev_gain, g->rec_X,
                                                         g->rec_y, g->rec_cap, g->rec_count);
  k_record_advance<<<1, 1, 0, g->stream>>>(&g->sctl->n_sel, g->rec_cap, g->rec_count);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

// Round-1 proposal (one CTA): the candidates list[0 .. *n_sel) (at most
// kProposeMax, the largest two-hop bounds) are scored by the network -- one
// warp per candidate, weights in shared memory -- and the kLanes with the
// largest predicted gain (ties: larger bound, then smaller id) are written
// back to list[0 .. 64) with *n_sel = min(64, count).  Only which candidates
// the first exact batch of round 1 holds changes; every other candidate is
// still compared with that batch's best exact gain by its bound.
constexpr int kProposeMax = 1024;
__global__ void __launch_bounds__(1024) k_round1_propose(int32_t *list, int32_t *n_sel, const float *__restrict__ W,
                                                        const int32_t *__restrict__ rp, const int32_t *__restrict__ dS,
                                                        const long long *__restrict__ ub,
                                                        const int32_t *__restrict__ stamp,
                                                        const long long *__restrict__ two_hop,
                                                        const int32_t *__restrict__ mx, long long prev_gain) {
  __shared__ float sw[kMlpParams];
  __shared__ float sh[32][kMlpHidden];
  __shared__ float s_key[kProposeMax];
  __shared__ long long s_ub[kProposeMax];
  __shared__ int s_id[kProposeMax];
  const int m = min(*n_sel, kProposeMax);
  for (int i = threadIdx.x; i < kMlpParams; i += blockDim.x) sw[i] = W[i];
  for (int i = threadIdx.x; i < kProposeMax; i += blockDim.x) {
    s_id[i] = i < m ? list[i] : INT_MAX;
    s_ub[i] = i < m ? ub[s_id[i]] : LLONG_MIN;
    s_key[i] = -INFINITY;
  }
  cta_sync();
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = wid; i < m; i += blockDim.x >> 5) {
    float f[kMlpIn];
    cand_features(s_id[i], rp, dS, ub, stamp, two_hop, mx, 1, prev_gain, f);
    const float o = mlp_forward_warp(sw, f, sh[wid]);
    if (lane == 0) s_key[i] = o;
  }
  cta_sync();
  // bitonic sort of (key desc, ub desc, id asc) over kProposeMax entries
  for (int size = 2; size <= kProposeMax; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      const int i = threadIdx.x, j = i ^ stride;
      if (j > i && i < kProposeMax) {
        const bool up = (i & size) == 0;  // this pair sorts "first = better"
        const bool ib = s_key[i] > s_key[j] || (s_key[i] == s_key[j] &&
                        (s_ub[i] > s_ub[j] || (s_ub[i] == s_ub[j] && s_id[i] < s_id[j])));
        if (ib != up) {
          const float tk = s_key[i]; s_key[i] = s_key[j]; s_key[j] = tk;
          const long long tu = s_ub[i]; s_ub[i] = s_ub[j]; s_ub[j] = tu;
          const int ti = s_id[i]; s_id[i] = s_id[j]; s_id[j] = ti;
        }
      }
      cta_sync();
    }
  }
  if (threadIdx.x < kLanes && threadIdx.x < m) list[threadIdx.x] = s_id[threadIdx.x];
  if (threadIdx.x == 0) *n_sel = min(m, kLanes);
}

int launch_round1_propose(gc_graph *g, long long prev_gain) {
  if (!g->prop_params) return GC_EINVAL;
  ++g->launches;
  k_round1_propose<<<1, 1024, 0, g->stream>>>(g->list, &g->sctl->n_sel, g->prop_params, g->rp, g->dS, g->ub,
                                              g->stamp, g->two_hop, g->mx, prev_gain);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

int launch_features(gc_graph *g, const int32_t *list, int32_t m, const int32_t *m_dev, int32_t round,
                    long long prev_gain, float *X) {
  ++g->launches;
  k_features<<<g->red_blocks, kRedThreads, 0, g->stream>>>(list, m, m_dev, g->rp, g->dS, g->ub, g->stamp,
                                                           g->two_hop, g->mx, round, prev_gain, X);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

// Gradient and loss into h->grad; lr > 0: and one Adam step.
static int mlp_grad_async(gc_mlp *h, const float *X, const float *y, int32_t m, float lr = 0.f) {
  const int tile = mlp_large(h, m) ? 64 : 16;
  const int ctas = (int)std::min<int64_t>(h->slots, ((int64_t)m + tile - 1) / tile);
  if (tile == 16)
    k_mlp_tile<1, true><<<ctas, kMlpThreads, mlp_smem(1), h->stream>>>(h->params, X, y, m, nullptr, h->part);
  else
    k_mlp_tile<4, true><<<ctas, kMlpThreads, mlp_smem(4), h->stream>>>(h->params, X, y, m, nullptr, h->part);
  const int blocks = (kMlpParams + 31) / 32;
  if (lr > 0) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    h->t += 1;
    const float c1 = 1.f - powf(b1, (float)h->t), c2 = 1.f - powf(b2, (float)h->t);
    k_mlp_reduce<true><<<blocks, kMlpThreads, 0, h->stream>>>(h->part, ctas, m, h->grad, h->params, h->adam_m,
                                                              h->adam_v, lr, b1, b2, eps, c1, c2);
  } else {
    k_mlp_reduce<false><<<blocks, kMlpThreads, 0, h->stream>>>(h->part, ctas, m, h->grad, nullptr, nullptr, nullptr,
                                                               0.f, 0.f, 0.f, 0.f, 0.f, 0.f);
  }
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

// Waits for gradient and loss on the host, through one pinned copy.
static int mlp_read_grad(gc_mlp *h, double *loss) {
  GC_CUDA(cudaMemcpyAsync(h->h_grad, h->grad, kMlpGradLen * sizeof(float), cudaMemcpyDeviceToHost, h->stream));
  GC_CUDA(cudaStreamSynchronize(h->stream));
  memcpy(loss, h->h_grad + kMlpLossAt, sizeof(double));
  return GC_OK;
}

}  // namespace gc

using namespace gc;

extern "C" {

int gc_mlp_create(int32_t max_batch, void *stream, gc_mlp **out) {
  if (!out || max_batch < 1) {
    set_error("bad argument to gc_mlp_create");
    return GC_EINVAL;
  }
  *out = nullptr;
  gc_mlp *h = new gc_mlp();
  h->max_batch = max_batch;
  h->stream = (cudaStream_t)stream;
  int dev = 0, sms = 0;
  bool ok = cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess;
  h->slots = kMlpCtasPerSm * sms;
  for (const void *f : {(const void *)k_mlp_tile<4, false>, (const void *)k_mlp_tile<4, true>})
    ok = ok &&
         cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mlp_smem(4)) == cudaSuccess;
  static_assert(mlp_smem(1) <= 48 * 1024, "needs no attribute");
  const size_t rows = (size_t)std::min<int64_t>(h->slots, ((int64_t)max_batch + 15) / 16);
  for (float **b : {&h->params, &h->adam_m, &h->adam_v})
    ok = ok && cudaMalloc((void **)b, kMlpParams * sizeof(float)) == cudaSuccess;
  ok = ok && cudaMalloc((void **)&h->grad, kMlpGradLen * sizeof(float)) == cudaSuccess &&
       cudaMalloc((void **)&h->part, rows * kMlpGradLen * sizeof(float)) == cudaSuccess &&
       cudaMallocHost((void **)&h->h_grad, kMlpGradLen * sizeof(float)) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    gc_mlp_free(h);
    set_error("gc_mlp_create: allocation failed");
    return GC_ENOMEM;
  }
  cudaMemsetAsync(h->params, 0, kMlpParams * sizeof(float), h->stream);
  cudaMemsetAsync(h->adam_m, 0, kMlpParams * sizeof(float), h->stream);
  cudaMemsetAsync(h->adam_v, 0, kMlpParams * sizeof(float), h->stream);
  *out = h;
  return GC_OK;
}

int gc_mlp_free(gc_mlp *h) {
  if (!h) return GC_OK;
  cudaStreamSynchronize(h->stream);
  void *bufs[] = {h->params, h->grad, h->adam_m, h->adam_v, h->part};
  for (void *b : bufs)
    if (b) cudaFree(b);
  if (h->h_grad) cudaFreeHost(h->h_grad);
  delete h;
  return GC_OK;
}

int gc_mlp_set_params(gc_mlp *h, const float *params) {
  if (!h || !params) {
    set_error("bad argument to gc_mlp_set_params");
    return GC_EINVAL;
  }
  GC_CUDA(cudaMemcpyAsync(h->params, params, kMlpParams * sizeof(float), cudaMemcpyHostToDevice, h->stream));
  GC_CUDA(cudaMemsetAsync(h->adam_m, 0, kMlpParams * sizeof(float), h->stream));
  GC_CUDA(cudaMemsetAsync(h->adam_v, 0, kMlpParams * sizeof(float), h->stream));
  h->t = 0;
  GC_CUDA(cudaStreamSynchronize(h->stream));
  return GC_OK;
}

int gc_mlp_get_params(gc_mlp *h, float *params) {
  if (!h || !params) {
    set_error("bad argument to gc_mlp_get_params");
    return GC_EINVAL;
  }
  GC_CUDA(cudaMemcpyAsync(params, h->params, kMlpParams * sizeof(float), cudaMemcpyDeviceToHost, h->stream));
  GC_CUDA(cudaStreamSynchronize(h->stream));
  return GC_OK;
}

int gc_mlp_forward(gc_mlp *h, const float *X, int32_t m, float *out) {
  if (!h || m < 0 || (m > 0 && (!X || !out))) {
    set_error("bad argument to gc_mlp_forward");
    return GC_EINVAL;
  }
  if (m == 0) return GC_OK;
  if (mlp_large(h, m)) {
    const int ctas = (int)std::min<int64_t>(h->slots, ((int64_t)m + 63) / 64);
    k_mlp_tile<4, false><<<ctas, kMlpThreads, mlp_smem(4), h->stream>>>(h->params, X, nullptr, m, out, nullptr);
  } else {
    k_mlp_forward<<<(m + 7) / 8, kMlpThreads, 0, h->stream>>>(h->params, X, m, out);
  }
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

int gc_mlp_grad(gc_mlp *h, const float *X, const float *y, int32_t m, float *grad, double *loss) {
  if (!h || !X || !y || m < 1 || m > h->max_batch) {
    set_error("bad argument to gc_mlp_grad (1 <= m <= max_batch)");
    return GC_EINVAL;
  }
  int rc = mlp_grad_async(h, X, y, m);
  if (rc) return rc;
  double l = 0;
  if ((rc = mlp_read_grad(h, &l))) return rc;
  if (grad) memcpy(grad, h->h_grad, kMlpParams * sizeof(float));
  if (loss) *loss = l;
  return GC_OK;
}

int gc_mlp_adam_step(gc_mlp *h, const float *X, const float *y, int32_t m, float lr) {
  if (!h || !X || !y || m < 1 || m > h->max_batch || !(lr > 0)) {
    set_error("bad argument to gc_mlp_adam_step");
    return GC_EINVAL;
  }
  return mlp_grad_async(h, X, y, m, lr);
}

int gc_mlp_train(gc_mlp *h, const float *X, const float *y, int32_t m, int32_t epochs, int32_t batch, float lr,
                 uint64_t seed, double *final_loss) {
  if (!h || !X || !y || m < 1 || epochs < 1 || batch < 1 || batch > h->max_batch || !(lr > 0)) {
    set_error("bad argument to gc_mlp_train");
    return GC_EINVAL;
  }
  const int32_t nb = (m + batch - 1) / batch;
  std::vector<int32_t> order(nb);
  uint64_t s = seed * 0x9E3779B97F4A7C15ULL + 1;
  for (int32_t e = 0; e < epochs; ++e) {
    for (int32_t i = 0; i < nb; ++i) order[i] = i;
    for (int32_t i = nb - 1; i > 0; --i) {  // Fisher-Yates on the minibatch order (xorshift64)
      s ^= s << 13;
      s ^= s >> 7;
      s ^= s << 17;
      std::swap(order[i], order[(int32_t)(s % (uint64_t)(i + 1))]);
    }
    for (int32_t i = 0; i < nb; ++i) {
      const int32_t off = order[i] * batch, len = std::min(batch, m - off);
      const int rc = mlp_grad_async(h, X + (size_t)off * kMlpIn, y + off, len, lr);
      if (rc) return rc;
    }
  }
  if (final_loss) {
    // loss over the whole set, one batch at a time
    double tot = 0;
    for (int32_t off = 0; off < m; off += batch) {
      const int32_t len = std::min(batch, m - off);
      double l = 0;
      int rc = mlp_grad_async(h, X + (size_t)off * kMlpIn, y + off, len);
      if (!rc) rc = mlp_read_grad(h, &l);
      if (rc) return rc;
      tot += l * len;
    }
    *final_loss = tot / m;
  }
  GC_CUDA(cudaStreamSynchronize(h->stream));
  return GC_OK;
}

int gc_candidate_features(const int32_t *row_ptr, const int32_t *dS, const int64_t *ub, const int32_t *stamp,
                          const int64_t *two_hop, const int32_t *mx, const int32_t *cand, int32_t m, int32_t round,
                          int64_t prev_gain, float *X, void *stream) {
  if (!row_ptr || !dS || !ub || !stamp || !two_hop || m < 0 || (m > 0 && (!cand || !X))) {
    set_error("bad argument to gc_candidate_features");
    return GC_EINVAL;
  }
  if (m == 0) return GC_OK;
  k_features<<<std::min(1024, (m + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
      cand, m, nullptr, row_ptr, dS, (const long long *)ub, stamp, (const long long *)two_hop, mx, round,
      (long long)prev_gain, X);
  GC_CUDA(cudaGetLastError());
  return GC_OK;
}

int gc_set_proposal(gc_graph *g, const gc_mlp *h, int32_t fill) {
  if (!g || fill < 0 || fill > kLanes - 1) {
    set_error("bad argument to gc_set_proposal (0 <= fill < 64)");
    return GC_EINVAL;
  }
  g->prop_params = h ? h->params : nullptr;
  g->prop_fill = h ? fill : 0;  // 0: round 1's first batch only
  return GC_OK;
}

int gc_set_recorder(gc_graph *g, float *X, float *y, int32_t cap) {
  if (!g || cap < 0 || (cap > 0 && (!X || !y))) {
    set_error("bad argument to gc_set_recorder");
    return GC_EINVAL;
  }
  g->rec_X = cap ? X : nullptr;
  g->rec_y = cap ? y : nullptr;
  g->rec_cap = cap;
  if (g->rec_count) GC_CUDA(cudaMemsetAsync(g->rec_count, 0, sizeof(int32_t), g->stream));
  return GC_OK;
}

int64_t gc_recorded(gc_graph *g) {
  if (!g || !g->rec_count) return -1;
  int32_t c = 0;
  if (cudaMemcpyAsync(&c, g->rec_count, sizeof(int32_t), cudaMemcpyDeviceToHost, g->stream) != cudaSuccess ||
      cudaStreamSynchronize(g->stream) != cudaSuccess)
    return -1;
  return c;
}

}  // extern "C"
