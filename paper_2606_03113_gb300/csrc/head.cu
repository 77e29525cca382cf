// head.cu -- statistics of the exit distributions P^(l) = softmax(z) (§3.1.1)
// from the logits that the LM-head product left in B.logits: maximum, argmax
// (lowest id on ties), top-8, log-sum-exp, entropy, token confidence.
//
// The product's own epilogue only scales and stores its logits (at most
// 128 KB to 0.5 MB a row against 131 MB to 1 GB of weights): statistics kept
// per tile there cost a merge of 152 blocks' parts per row at the end of the
// launch, one row after the other (13 rows of a 128256-token vocabulary: 200
// us more in a verification pass).  Here a grid of (vocabulary chunks, rows)
// reads them back from L2, and the last chunk of a row merges the row's
// parts, so all rows end together: 6 us, bound by the chain of block
// barriers and the round trips of the row's ticket.
//
// Every sum has a fixed order that depends on the vocabulary alone, so a
// row's statistics are the same whatever the number of rows.  A NaN or -inf
// logit takes part in nothing; a +inf one is the maximum, and the sums (lse,
// entropy, pmax, C_k) are NaN, so that no draw is made from such a row.
#include <math.h>

#include "kernels.h"
#include "pipe.cuh"

namespace ssd {

namespace {

constexpr int kHThreads = 256;
constexpr int kHPer = 8;                          // logits per thread and chunk
constexpr int kHChunk = kHThreads * kHPer;
constexpr int kHWarps = kHThreads / 32;

// (value, id) as one key: larger values first, then lower ids.  0: none.
struct Key {
  uint32_t hi, lo;
};

__device__ __forceinline__ Key make_key(float z, int id) {
  if (!(z > -INFINITY)) return Key{0u, 0u};  // -inf and NaN take part in nothing
  const uint32_t b = __float_as_uint(z + 0.f);
  return Key{b & 0x80000000u ? ~b : b | 0x80000000u, ~(uint32_t)id};
}
__device__ __forceinline__ bool key_less(Key a, Key b) {
  return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
}
__device__ __forceinline__ float key_value(Key k) {
  if (!k.hi) return -INFINITY;
  return __uint_as_float(k.hi & 0x80000000u ? k.hi ^ 0x80000000u : ~k.hi);
}
__device__ __forceinline__ int key_id(Key k) { return k.hi ? (int)~k.lo : 0x7fffffff; }

struct HeadSmem {
  Key warp_top[kHWarps][kTopK];
  Key top[kTopK];
  float f[kHWarps];
  int last;
};

// The warp's kTopK largest of its lanes' N keys each, in order; lane r < kTopK
// returns the r-th.  The keys are used up.
template <int N>
__device__ __forceinline__ Key warp_topk(Key (&k)[N], int lane) {
  Key best = k[0], mine{0u, 0u};
#pragma unroll
  for (int i = 1; i < N; ++i)
    if (key_less(best, k[i])) best = k[i];
#pragma unroll
  for (int r = 0; r < kTopK; ++r) {
    const uint32_t hi = __reduce_max_sync(0xffffffffu, best.hi);
    const uint32_t lo = __reduce_max_sync(0xffffffffu, best.hi == hi ? best.lo : 0u);
    if (lane == r) mine = Key{hi, lo};
    if (hi && best.hi == hi && best.lo == lo) {
      Key nb{0u, 0u};
#pragma unroll
      for (int i = 0; i < N; ++i) {
        if (k[i].hi == hi && k[i].lo == lo) k[i] = Key{0u, 0u};
        if (key_less(nb, k[i])) nb = k[i];
      }
      best = nb;
    }
  }
  return mine;
}

// The block's kTopK largest keys into sm.top (visible to the whole block).
template <int N>
__device__ __forceinline__ void block_topk(Key (&k)[N], HeadSmem& sm) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Key w = warp_topk(k, lane);
  if (lane < kTopK) sm.warp_top[warp][lane] = w;
  __syncthreads();
  if (warp == 0) {
    const Key* all = &sm.warp_top[0][0];
    Key c[2] = {all[lane], all[lane + 32]};
    static_assert(kHWarps * kTopK == 64, "two keys per lane");
    const Key t = warp_topk(c, lane);
    if (lane < kTopK) sm.top[lane] = t;
  }
  __syncthreads();
}

__device__ __forceinline__ float block_max(float v, HeadSmem& sm) {
  v = warp_max(v);
  if ((threadIdx.x & 31) == 0) sm.f[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = sm.f[0];
#pragma unroll
  for (int w = 1; w < kHWarps; ++w) r = fmaxf(r, sm.f[w]);
  __syncthreads();
  return r;
}

__device__ __forceinline__ float block_sum(float v, HeadSmem& sm) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) sm.f[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = 0.f;
#pragma unroll
  for (int w = 0; w < kHWarps; ++w) r += sm.f[w];
  __syncthreads();
  return r;
}

}  // namespace

// Grid (chunks of kHChunk logits, at most kHeadParts of them; rows).
__global__ void __launch_bounds__(kHThreads) k_head_stats(const Dims D, const Bufs B, RowSel sel,
                                                          int topk) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ HeadSmem sm;
  int pos0, M;
  resolve_rows(B.ctl, sel, pos0, M);
  const int m = blockIdx.y, tid = threadIdx.x;
  if (m >= M) return;
  const float* z = B.logits + (size_t)m * D.V;
  const int nchunks = (D.V + kHChunk - 1) / kHChunk;

  float mx = -INFINITY, S = 0.f, T = 0.f;  // of the block's chunks so far
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const int v0 = c * kHChunk;
    float x[kHPer];
    Key k[kHPer + 1];
#pragma unroll
    for (int j = 0; j < kHPer; ++j) {
      const int v = v0 + j * kHThreads + tid;
      x[j] = v < D.V ? __ldcg(z + v) : -INFINITY;
    }
    float tm = -INFINITY;
#pragma unroll
    for (int j = 0; j < kHPer; ++j) {
      k[j] = make_key(x[j], v0 + j * kHThreads + tid);
      tm = fmaxf(tm, k[j].hi ? x[j] : -INFINITY);
    }
    k[kHPer] = c != (int)blockIdx.x && tid < kTopK ? sm.top[tid] : Key{0u, 0u};
    const float cm = block_max(tm, sm);
    float s = 0.f, t = 0.f;
#pragma unroll
    for (int j = 0; j < kHPer; ++j)
      if (k[j].hi) {
        const float d = x[j] - cm, e = expf(d);
        s += e;
        t = fmaf(e, d, t);
      }
    s = block_sum(s, sm);
    t = block_sum(t, sm);
    // (a sum that is not a number, from an infinite logit, stays one)
    if (S != 0.f && s != 0.f) {
      const float nm = fmaxf(mx, cm), ea = expf(mx - nm), eb = expf(cm - nm);
      T = ea * (T + (mx - nm) * S) + eb * (t + (cm - nm) * s);
      S = S * ea + s * eb;
      mx = nm;
    } else if (s != 0.f) {
      mx = cm;
      S = s;
      T = t;
    }
    block_topk(k, sm);
  }

  HeadPart* parts = static_cast<HeadPart*>(B.head_part) + (size_t)m * kHeadParts;
  const int np = gridDim.x;
  if (np > 1) {
    HeadPart* mine = parts + blockIdx.x;
    if (tid == 0) {
      mine->mx = mx;
      mine->S = S;
      mine->T = T;
    }
    if (tid < kTopK) {
      mine->tv[tid] = key_value(sm.top[tid]);
      mine->ti[tid] = key_id(sm.top[tid]);
    }
    __syncthreads();
    if (tid == 0) sm.last = atom_add_acq_rel_gpu(B.head_counter + m, 1u) == (uint32_t)(np - 1);
    __syncthreads();
    if (!sm.last) return;
    // the row's last block: parts b = tid, tid + 256, ... per thread
    static_assert(kHeadParts == kHThreads, "one part per thread");
    float pm = -INFINITY, ps = 0.f, pt = 0.f;
    if (tid < np) {
      pm = __ldcg(&parts[tid].mx);
      ps = __ldcg(&parts[tid].S);
      pt = __ldcg(&parts[tid].T);
    }
    Key k[kTopK];
#pragma unroll
    for (int j = 0; j < kTopK; ++j) {
      const int i = j * kHThreads + tid;  // candidate i: entry i % 8 of part i / 8
      const HeadPart* p = parts + (i >> 3);
      k[j] = i < np * kTopK ? make_key(__ldcg(&p->tv[i & 7]), __ldcg(&p->ti[i & 7])) : Key{0u, 0u};
    }
    mx = block_max(ps != 0.f ? pm : -INFINITY, sm);
    const float d = pm - mx, e = ps != 0.f ? expf(d) : 0.f;
    S = block_sum(ps != 0.f ? ps * e : 0.f, sm);
    T = block_sum(ps != 0.f ? e * (pt + d * ps) : 0.f, sm);
    block_topk(k, sm);
    if (tid == 0) B.head_counter[m] = 0u;
  }
  if (tid == 0) {
    // H = log S - T / S, C_k = lse - mean of the k largest logits, pmax = 1 / S
    RowStats& o = B.stats[m];
    const float logS = logf(S);
    o.argmax = key_id(sm.top[0]);
    o.zmax = mx;
    o.lse = mx + logS;
    o.entropy = logS - T / S;
    float tsum = 0.f;
#pragma unroll
    for (int q = 0; q < kTopK; ++q) {
      const float v = key_value(sm.top[q]);
      o.top_idx[q] = key_id(sm.top[q]);
      o.top_logit[q] = v;
      if (q < topk) tsum += v;
    }
    o.conf_k = o.lse - tsum / (float)topk;
    o.pmax = 1.0f / S;
    o.margin = key_value(sm.top[0]) - key_value(sm.top[1]);
  }
}

cudaError_t launch_head_stats(const Dims& D, const Bufs& B, int topk, RowSel sel, int mrows,
                              cudaStream_t st) {
  const int nchunks = (D.V + kHChunk - 1) / kHChunk;
  const dim3 grid(nchunks < kHeadParts ? nchunks : kHeadParts, mrows);
  return launch_ex(k_head_stats, grid, dim3(kHThreads), 0, st, D, B, sel, topk);
}

}  // namespace ssd
