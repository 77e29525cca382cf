// fp32.cu -- matrix-vector kernels of fp32 decoders: QKV, O, gate/up, down and
// the exit head for M <= 17 input rows.
//
// The fp32 decoders are small ones: a pass is a chain of short kernels whose
// weights stay in L2.  So each kernel is a single pass without shared memory,
// rings or block barriers: a warp owns a pair of rows (the pair that the
// epilogue combines), holds 512 columns of both in registers, the first of
// them loaded before the wait for the previous kernel, and multiplies them
// with all M input rows (read through L1).  RMSNorm needs no sums from the
// kernel that wrote the rows: the warp reads whole rows anyway and adds their
// squares beside the products.
//
// Bound by the launch and two dependent round trips to L2 in a small model, by
// HBM in a large one.  us for one pass of 1 / 5 / 17 rows, through L layers and
// the head (4 d tokens, FFN 2.7 d, 40 tokens of context), against the streamed
// kernels (persistent blocks, shared-memory ring, row tiles split over blocks
// and joined again) that did this before:
//   d = 256, L = 4:   129 /  165 /  298   (332 /  521 /  905)
//   d = 1024, L = 4:  180 /  259 /  493   (408 /  730 / 1402)
//   d = 4096, L = 1:  242 /  367 /  842   (293 /  900 / 2116)
//   d = 8192, L = 1:  735 / 1144 / 2610   (755 / 2780 / 6841)
// so these kernels serve every size.
#include <math.h>

#include "kernels.h"
#include "pipe.cuh"

namespace ssd {

namespace {

constexpr int kSWarps = 4;
constexpr int kSChunk = 512;             // columns in registers: four float4 a lane and row
constexpr int kSVec = kSChunk / 128;
constexpr int kSRows = 4;                // input rows whose loads are in flight together

enum SKind : int { kSQkv = 0, kSGateUp = 1, kSResid = 2, kSHead = 3 };

struct SArgs {
  Dims D;
  Bufs B;
  const float* W;
  const float* gnorm;  // RMSNorm weights of the input (NORM)
  const float* x;      // [M][K]
  int N, K;
  int layer;
  RowSel sel;
};

// First and second row of pair p.
template <int KIND>
__device__ __forceinline__ void pair_rows(const SArgs& a, int p, int& r0, int& r1) {
  if constexpr (KIND == kSQkv) {
    const int half = a.D.hd / 2, head = p / half;
    r0 = head * a.D.hd + (p - head * half);
    r1 = r0 + half;
  } else if constexpr (KIND == kSGateUp) {
    r0 = p;
    r1 = a.N / 2 + p;
  } else {
    r0 = 2 * p;
    r1 = r0 + 1;
  }
}

template <int MM>
__device__ __forceinline__ float pick_lane(const float (&v)[MM], int lane) {
  float r = 0.f;
#pragma unroll
  for (int m = 0; m < MM; ++m)
    if (m == lane) r = v[m];
  return r;
}

__device__ __forceinline__ float4 weights4(const float* p) {
  const uint4 u = ld_stream16(p);
  return make_float4(__uint_as_float(u.x), __uint_as_float(u.y), __uint_as_float(u.z),
                     __uint_as_float(u.w));
}

}  // namespace

template <int KIND, int MM>
__global__ void __launch_bounds__(kSWarps * 32) k_rows_f32(const SArgs a) {
  constexpr bool NORM = KIND != kSResid;
  pdl_launch_dependents();
  const Dims& D = a.D;
  const int lane = threadIdx.x & 31;
  const int p = blockIdx.x * kSWarps + (threadIdx.x >> 5);
  const bool live = p < a.N / 2;
  int r0, r1;
  pair_rows<KIND>(a, live ? p : 0, r0, r1);
  const float* w0 = a.W + (size_t)r0 * a.K + 4 * lane;
  const float* w1 = a.W + (size_t)r1 * a.K + 4 * lane;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  // a chunk of both rows and of the norm weights; with few input rows the
  // next chunk is loaded while this one is multiplied (one row, d = 8192: 735
  // us against 876; with kMaxM rows the registers are needed for their sums)
  constexpr bool kAhead = MM <= 8;
  struct Chunk {
    float4 a[kSVec], b[kSVec], g[NORM ? kSVec : 1];
  };
  Chunk cur, next;
  auto load = [&](Chunk& c, int k0) {
#pragma unroll
    for (int j = 0; j < kSVec; ++j) {
      const int k = k0 + 128 * j;
      const bool in = k + 4 * lane < a.K;
      c.a[j] = in ? weights4(w0 + k) : zero;
      c.b[j] = in ? weights4(w1 + k) : zero;
      if constexpr (NORM)
        c.g[j] = in ? __ldg(reinterpret_cast<const float4*>(a.gnorm + k + 4 * lane)) : zero;
    }
  };
  load(cur, 0);
  pdl_wait();
  int pos0, M;
  resolve_rows(a.B.ctl, a.sel, pos0, M);
  if (M > MM) M = MM;  // the launcher picks MM >= M
  if (!live) return;

  float s0[MM], s1[MM], sq[NORM ? MM : 1];
#pragma unroll
  for (int m = 0; m < MM; ++m) {
    s0[m] = s1[m] = 0.f;
    if (NORM) sq[m] = 0.f;
  }
  // four columns each, then pairs: short chains, small errors
  auto dot = [&](const float4 (&u)[kSVec], const float4 (&v)[kSVec]) -> float {
    float q[kSVec];
#pragma unroll
    for (int j = 0; j < kSVec; ++j)
      q[j] = fmaf(u[j].w, v[j].w, fmaf(u[j].z, v[j].z, fmaf(u[j].y, v[j].y, u[j].x * v[j].x)));
    static_assert(kSVec == 4, "two levels of pairs");
    return (q[0] + q[1]) + (q[2] + q[3]);
  };
  for (int k0 = 0; k0 < a.K; k0 += kSChunk) {
    if (!kAhead && k0) load(cur, k0);
    if (kAhead && k0 + kSChunk < a.K) load(next, k0 + kSChunk);
    if constexpr (NORM) {
#pragma unroll
      for (int j = 0; j < kSVec; ++j) {
        const float4 g = cur.g[j];
        cur.a[j] = make_float4(cur.a[j].x * g.x, cur.a[j].y * g.y, cur.a[j].z * g.z, cur.a[j].w * g.w);
        cur.b[j] = make_float4(cur.b[j].x * g.x, cur.b[j].y * g.y, cur.b[j].z * g.z, cur.b[j].w * g.w);
      }
    }
    // kSRows rows at a time: their loads are in flight together
#pragma unroll
    for (int mb = 0; mb < MM; mb += kSRows) {
      if (mb >= M) break;
      float4 x[kSRows][kSVec];
#pragma unroll
      for (int r = 0; r < kSRows; ++r)
#pragma unroll
        for (int j = 0; j < kSVec; ++j)
          x[r][j] = mb + r < M && k0 + 128 * j + 4 * lane < a.K
                        ? *reinterpret_cast<const float4*>(a.x + (size_t)(mb + r) * a.K + k0 +
                                                           128 * j + 4 * lane)
                        : zero;
#pragma unroll
      for (int r = 0; r < kSRows; ++r) {
        if (mb + r >= MM) continue;
        constexpr int kLast = MM - 1;
        const int m = mb + r < kLast ? mb + r : kLast;
        s0[m] += dot(cur.a, x[r]);
        s1[m] += dot(cur.b, x[r]);
        if (NORM) sq[m] += dot(x[r], x[r]);
      }
    }
    if (kAhead) cur = next;
  }
#pragma unroll
  for (int m = 0; m < MM; ++m)
    if (m < M) {
      s0[m] = warp_sum(s0[m]);
      s1[m] = warp_sum(s1[m]);
      if (NORM) sq[m] = warp_sum(sq[m]);
    }
  // lane m finishes row m
  const int t = lane;
  if (t >= M) return;
  float y0 = pick_lane(s0, t), y1 = pick_lane(s1, t);
  if constexpr (NORM) {
    const float rs = 1.0f / sqrtf(pick_lane(sq, t) / (float)a.K + D.eps);
    y0 *= rs;
    y1 *= rs;
  }
  if constexpr (KIND == kSResid) {
    float* h = a.B.h + (size_t)t * D.d;
    h[r0] = __ldcg(h + r0) + y0;
    h[r1] = __ldcg(h + r1) + y1;
  } else if constexpr (KIND == kSHead) {
    float* z = a.B.logits + (size_t)t * D.V;
    z[r0] = y0;
    z[r1] = y1;
  } else if constexpr (KIND == kSGateUp) {
    a.B.act[(size_t)t * D.F + p] = y0 / (1.0f + expf(-y0)) * y1;
  } else {
    const int half = D.hd / 2, head = p / half, i = p - head * half, pos = pos0 + t;
    float* kv = static_cast<float*>(a.B.kv) + (size_t)a.layer * 2 * D.Hkv * D.max_seq * D.hd;
    float* out;
    if (head < D.Hq + D.Hkv) {
      // rotary embedding (angle pos * theta^(-2i/hd) from the table)
      const float2 cs = a.B.rope[(size_t)pos * half + i];
      const float o0 = y0 * cs.x - y1 * cs.y, o1 = y1 * cs.x + y0 * cs.y;
      y0 = o0;
      y1 = o1;
      out = head < D.Hq ? a.B.xq + (size_t)t * D.qd + (size_t)head * D.hd
                        : kv + ((size_t)(head - D.Hq) * D.max_seq + pos) * D.hd;
    } else {
      out = kv + ((size_t)(head - D.Hq) * D.max_seq + pos) * D.hd;  // Hkv + value head
    }
    out[i] = y0;
    out[i + half] = y1;
  }
}

namespace {

template <int KIND>
cudaError_t rows_launch(const SArgs& a, int mrows, cudaStream_t st) {
  const dim3 grid((a.N / 2 + kSWarps - 1) / kSWarps), blk(kSWarps * 32);
  if (mrows == 1) return launch_ex(k_rows_f32<KIND, 1>, grid, blk, 0, st, a);
  if (mrows <= 8) return launch_ex(k_rows_f32<KIND, 8>, grid, blk, 0, st, a);
  return launch_ex(k_rows_f32<KIND, kMaxM>, grid, blk, 0, st, a);
}

}  // namespace

// Part 0 (QKV), 2 (O), 3 (gate/up) or 4 (down) of a layer.
cudaError_t launch_f32_part(const Dims& D, const Bufs& B, const LayerW& w, int layer, int part,
                              RowSel sel, int mrows, cudaStream_t st) {
  SArgs a{};
  a.D = D;
  a.B = B;
  a.sel = sel;
  a.layer = layer;
  switch (part) {
    case 0:
      a.N = (D.Hq + 2 * D.Hkv) * D.hd;
      a.K = D.d;
      a.W = static_cast<const float*>(w.wqkv);
      a.gnorm = static_cast<const float*>(w.attn_norm);
      a.x = B.h;
      return rows_launch<kSQkv>(a, mrows, st);
    case 2:
      a.N = D.d;
      a.K = D.qd;
      a.W = static_cast<const float*>(w.wo);
      a.x = B.attn_out;
      return rows_launch<kSResid>(a, mrows, st);
    case 3:
      a.N = 2 * D.F;
      a.K = D.d;
      a.W = static_cast<const float*>(w.wgu);
      a.gnorm = static_cast<const float*>(w.ffn_norm);
      a.x = B.h;
      return rows_launch<kSGateUp>(a, mrows, st);
    case 4:
      a.N = D.d;
      a.K = D.F;
      a.W = static_cast<const float*>(w.wdown);
      a.x = B.act;
      return rows_launch<kSResid>(a, mrows, st);
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_f32_head(const Dims& D, const Bufs& B, const void* lm, const void* final_norm,
                              RowSel sel, int mrows, cudaStream_t st) {
  SArgs a{};
  a.D = D;
  a.B = B;
  a.sel = sel;
  a.N = D.V;
  a.K = D.d;
  a.W = static_cast<const float*>(lm);
  a.gnorm = static_cast<const float*>(final_norm);
  a.x = B.h;
  return rows_launch<kSHead>(a, mrows, st);
}

}  // namespace ssd
