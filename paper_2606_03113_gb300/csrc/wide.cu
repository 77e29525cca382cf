// wide.cu -- prompt processing of the bf16 decoder (sm_103a): up to kWideCap
// prompt rows per pass through all layers, so that a weight is read once per
// chunk of the prompt and not once per 16 rows.
//
// Products (k_wide): C[token][row] = sum_k W[row][k] x[token][k] on the
// 5th-generation tensor cores.  A tile is 128 weight rows x TT tokens; the
// input rows enter as bf16 high and low parts (x = hi + lo to 16 significant
// bits, the split of the decode kernels), which stand side by side as one
// operand of N = 2 TT columns, so one weight tile in shared memory serves
// both.  The kernel that produces an input row writes its two parts already
// multiplied by the RMSNorm weights of the product that reads it; the
// norm's scale is applied to the product (per-tile sums of squares travel
// beside the rows).
//  - a product with fewer tiles than SMs (a short prompt's O and down) splits K
//    over up to eight blocks per tile, whose last one adds their sums.  How K
//    is cut into groups and segments, and the order of their sums, depends on the
//    matrix and the device alone, so a row's bits do not depend on the length of
//    the prompt;
//  - persistent grid, tiles dealt round robin with the token tiles of one
//    weight tile next to each other (they share it in L2);
//  - warp roles (320 threads): a TMA warp fills a ring of 64-column stages
//    (two 64 x 64 weight boxes, one hi/lo input box), one thread issues
//    tcgen05.mma (M = 128, N = 2 TT, K = 16) into double-buffered TMEM
//    accumulators, eight warps run the fused epilogue of one tile while the
//    next one multiplies;
//  - a rotary or gate/up pair of a tile sits in rows r and r + 64, that is in
//    TMEM lanes of different warps: they swap halves through shared memory.
// Bound by the tensor cores and by the copies out of L2 (48 KB per stage of
// a 128-token tile in 512 cycles of tcgen05.mma at full rate).  512 rows of
// the Llama-2-7B shape: gate/up 122 us (1.51 PFLOP/s with both parts), QKV 84,
// down 75, O 38 us.  In passes of 16 rows through the decode kernels a 508-token
// prompt through four layers and its last rows' logits took 18.8 ms, in chunks
// 2.2 ms; 2043 tokens of the 13B shape 105 ms and 9.8 ms.  The exit head of a
// prompt's last rows (20 of them feed the C_trace window) is such a product
// too, one pass over the LM head instead of one per 16 rows: that took a
// 93-token prompt of the 8B widths (4 layers, 128256 tokens) from 2188 to 1912
// us, splitting K then to 1740.
// Attention (k_attn_wide): 64 query rows x one head per block, 64-key steps
// with a running maximum; scores and outputs on mma.sync with the fp32
// operand (queries, probabilities) in three bf16 parts, 24 bits, so nothing
// is rounded below fp32.  Bound by mma.sync: 512 rows of the Llama-2-7B shape
// take 42 us a layer, rows 1024-1919 of the 13B shape 252 us (328 TFLOP/s with
// the three parts).
#include <math.h>

#include <algorithm>

#include "kernels.h"
#include "mma.cuh"
#include "pipe.cuh"
#include "tc.cuh"

namespace ssd {

namespace {

constexpr int kWR = 128;              // weight rows per tile
constexpr int kWK = 64;               // columns per stage
constexpr int kWEpi = 8;              // epilogue warps
constexpr int kWEThreads = kWEpi * 32;
constexpr int kWTmaWarp = kWEpi, kWMmaWarp = kWEpi + 1;
constexpr int kWThreads = (kWEpi + 2) * 32;
constexpr int kWChunk = 16;           // tokens per epilogue step of a warp
// K is summed in segments of at most this many stages, one TMEM accumulator
// each, which the epilogue warps add in their registers: the tensor core's
// running sum is cut and not rounded at each 16-column step, so a sum over all
// of K in TMEM would be off by up to K / 16 units in the last place, to one
// side.  1024 columns at a time keep that at 64, as in the decode kernels, whose
// blocks sum 450 to 2300 columns of a row each.  The drain is hidden by the
// other accumulator but for its own tensor-memory reads: 512 tokens of the
// 12288 x 4096 product take 83.7 us (94.5 us with 512 columns at a time, 76.5 us
// with all of K).
constexpr int kWSeg = 16;

enum WKind : int { kWQkv = 0, kWResid = 1, kWGateUp = 2, kWHead = 3 };
// O and down are the products that short prompts split most and over the longest
// K: their segments are added in groups first, so that a split leaves few sums to
// join (down of the 8B shape, 89 rows: 4 a tile instead of 13, 41.5 us against
// 48.4; a second accumulator costs the others 1 % of a long prompt).
constexpr bool w_grouped(int kind) { return kind == kWResid; }

template <int TT>
struct WL {
  static constexpr int N = 2 * TT;
  static constexpr int A = kWR * kWK * 2;
  static constexpr int X = N * kWK * 2;
  static constexpr int Stage = A + X;
  static constexpr int NS = TT == 128 ? 4 : (TT == 64 ? 6 : 8);
  static constexpr uint32_t kCols = 2 * N;
  static constexpr size_t exch = (size_t)NS * Stage;                  // [2][warps][8][32] floats
  static constexpr size_t rs = exch + 2 * kWEpi * 8 * 32 * 4;          // [TT]
  static constexpr size_t red = rs + TT * 4;                           // [4][TT]
  static constexpr size_t bars = red + 4 * TT * 4;                     // full, empty, accfull, accempty
  static constexpr size_t tslot = bars + 8 * (2 * NS + 4);
  static constexpr size_t total = tslot + 16 + 1024;
  static_assert(total <= 227 * 1024, "shared memory budget");
};

struct WArgs {
  Dims D;
  Bufs B;
  WideBufs P;
  int N, K, nks, nrt, ntt;     // rows, columns, stages, row tiles, token tiles
  int ngrp, spg;               // groups of K, segments of a group (1 but for grouped kinds)
  int seg_q, seg_r;            // stages of a segment; the first seg_r have one more
  int nsp;                     // parts that K is split into (blocks that share a tile)
  int M, pos0, layer;
  int row0;                    // first of the M input rows
  const float* ss_in;          // per-tile sums of squares of the input rows, or null
  float* ss_out;               // residual: the same for the rows written
  const __nv_bfloat16* gnext;  // residual: norm weights of the next product (null: none)
};

// First stage of segment g of K.
__device__ __forceinline__ int w_seg_start(const WArgs& a, int g) {
  return g * a.seg_q + min(g, a.seg_r);
}

// Work item `it`: row tile, token tile and part of K (groups g0 .. g1 - 1,
// stages k0 .. k0 + n - 1).
struct WItem {
  int rt, tt, sp, g0, g1, k0, n;
  __device__ WItem(const WArgs& a, int it) {
    tt = it % a.ntt;
    const int r = it / a.ntt;
    sp = r % a.nsp;
    rt = r / a.nsp;
    g0 = a.ngrp * sp / a.nsp;
    g1 = a.ngrp * (sp + 1) / a.nsp;
    k0 = w_seg_start(a, g0 * a.spg);
    n = w_seg_start(a, g1 * a.spg) - k0;
  }
};

// Partial sums that the parts of a tile leave: one of the first part, whose
// groups are the first terms of the sum over K, and one of each later group.
__host__ __device__ inline int w_slots(int ngrp, int nsp) { return ngrp - ngrp / nsp + 1; }

__device__ __forceinline__ void w_flag(const Bufs& B) { atomicOr(&B.ctl->err, (int)kErrTimeout); }

__device__ __forceinline__ void tma_load_2d_plain(void* dst, const CUtensorMap* map, int c0, int r0,
                                                  uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(r0), "r"(smem_u32(bar))
      : "memory");
}

// 8 or 16 columns of the warp's TMEM lanes from two places (high and low parts),
// added.
__device__ __forceinline__ void tc_ld_sum(uint32_t hi, uint32_t lo, float (&v)[8]) {
  uint32_t a[8], b[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]),
                 "=r"(a[7])
               : "r"(hi)
               : "memory");
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]),
                 "=r"(b[7])
               : "r"(lo)
               : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(a[i]) + __uint_as_float(b[i]);
}
__device__ __forceinline__ void tc_ld_sum(uint32_t hi, uint32_t lo, float (&v)[16]) {
  uint32_t a[16], b[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];"
      : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]),
        "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]),
        "=r"(a[14]), "=r"(a[15])
      : "r"(hi)
      : "memory");
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];"
      : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]),
        "=r"(b[7]), "=r"(b[8]), "=r"(b[9]), "=r"(b[10]), "=r"(b[11]), "=r"(b[12]), "=r"(b[13]),
        "=r"(b[14]), "=r"(b[15])
      : "r"(lo)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(a[i]) + __uint_as_float(b[i]);
}

// Sums of 16 values over the warp's 32 lanes in a fixed order; lane 2 i (and
// 2 i + 1) returns the sum of value i.
__device__ __forceinline__ float warp_sum16(float (&v)[16], int lane) {
#pragma unroll
  for (int off = 16, n = 8; n >= 1; off >>= 1, n >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i < n) {
        const float keep = up ? v[i + n] : v[i], give = up ? v[i] : v[i + n];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
      }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

}  // namespace

template <int TT, int KIND>
__global__ void __launch_bounds__(kWThreads, 1)
    k_wide(const __grid_constant__ CUtensorMap wmap, const __grid_constant__ CUtensorMap xmap,
           const WArgs a) {
  using S = WL<TT>;
  constexpr int NS = S::NS, N = S::N;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::bars);
  uint64_t* empty = full + NS;
  uint64_t* accfull = empty + NS;
  uint64_t* accempty = accfull + 2;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + S::tslot);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  if (tid == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&accfull[i], 1);
      mbar_init(&accempty[i], kWEpi);
    }
    mbar_init_fence();
  }
  if (warp == kWMmaWarp) tc_alloc(tslot, S::kCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  __shared__ int s_last;
  pdl_launch_dependents();

  const int ntiles = a.nrt * a.ntt * a.nsp;
  if (warp == kWTmaWarp) {
    if (lane == 0) {
      tma_prefetch_desc(&wmap);
      tma_prefetch_desc(&xmap);
      // weight boxes of the first stages need nothing from earlier kernels
      auto weights = [&](int slot, int rt, int kc) {
        unsigned char* dst = smem + (size_t)slot * S::Stage;
        mbar_arrive_expect_tx(&full[slot], (uint32_t)S::Stage);
        const int r0 = KIND == kWGateUp ? rt * 64 : rt * 128;
        const int r1 = KIND == kWGateUp ? a.N / 2 + rt * 64 : rt * 128 + 64;
        tma_load_2d_plain(dst, &wmap, kc * kWK, r0, &full[slot]);
        tma_load_2d_plain(dst + S::A / 2, &wmap, kc * kWK, r1, &full[slot]);
      };
      bool ok = true;
      int npre = 0;
      if ((int)blockIdx.x < ntiles) {
        const WItem w(a, blockIdx.x);
        for (; npre < NS && npre < w.n; ++npre) weights(npre, w.rt, w.k0 + npre);
      }
      pdl_wait();
      asm volatile("fence.proxy.async.global;" ::: "memory");
      int slot = 0, it = 0;
      uint32_t ph = 1;
      for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        const WItem w(a, tile);
        for (int i = 0; i < w.n; ++i, ++it) {
          const int kc = w.k0 + i;
          if (it >= npre) {
            if (!mbar_wait(&empty[slot], ph)) {
              ok = false;
              break;
            }
            weights(slot, w.rt, kc);
          }
          tma_load_3d(smem + (size_t)slot * S::Stage + S::A, &xmap, kc * kWK, a.row0 + w.tt * TT, 0, &full[slot]);
          if (++slot == NS) {
            slot = 0;
            ph ^= 1u;
          }
        }
      }
      if (!ok) w_flag(a.B);
      // every copy has landed before the block exits
      for (int j = it > NS ? it - NS : 0; j < it; ++j) mbar_wait(&full[j % NS], (uint32_t)(j / NS) & 1u);
    }
  } else if (warp == kWMmaWarp) {
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(128, N);
      bool ok = true;
      int slot = 0, sc = 0;
      uint32_t ph = 0;
      for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        const WItem w(a, tile);
        int sg = w.g0 * a.spg, seg_end = w_seg_start(a, sg + 1);
        bool first = true;
        for (int kc = w.k0; kc < w.k0 + w.n; ++kc) {
          if (first && !(ok = mbar_wait(&accempty[sc & 1], ((uint32_t)(sc >> 1) & 1u) ^ 1u))) break;
          if (!(ok = mbar_wait(&full[slot], ph))) break;
          tc_fence_after();
          const uint32_t d = tmem + (uint32_t)((sc & 1) * N);
          const uint32_t ab = smem_u32(smem + (size_t)slot * S::Stage);
          const uint32_t xb = ab + S::A;
#pragma unroll
          for (int kk = 0; kk < kWK / 16; ++kk)
            tc_mma_bf16(d, sdesc_k128(ab + kk * 32), sdesc_k128(xb + kk * 32), idesc,
                        !first || kk > 0);
          tc_commit(&empty[slot]);
          first = kc + 1 == seg_end;
          if (first) {
            tc_commit(&accfull[sc++ & 1]);
            seg_end = w_seg_start(a, ++sg + 1);
          }
          if (++slot == NS) {
            slot = 0;
            ph ^= 1u;
          }
        }
      }
      if (!ok) w_flag(a.B);
    }
  } else {
    // ---------------- epilogue warps: lane quarter q, token half th
    pdl_wait();
    float* exch = reinterpret_cast<float*>(smem + S::exch);
    float* srs = reinterpret_cast<float*>(smem + S::rs);
    float* red = reinterpret_cast<float*>(smem + S::red);
    const Dims& D = a.D;
    const int q = warp & 3, th = warp >> 2;
    bool ok = true;
    int sc = 0, xp = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
      const WItem w(a, tile);
      const int rt = w.rt, t0 = w.tt * TT;
      if constexpr (KIND != kWResid) {
        // RMSNorm scale of the tile's input rows: their sums of squares per
        // 128 columns, added in column order
        for (int t = tid; t < TT; t += kWEThreads) {
          float sum = 0.f;
          if (t0 + t < a.M) {
            const float* sp = a.ss_in + t0 + t;
            const int np = (a.K + kWR - 1) / kWR;
#pragma unroll 8
            for (int c = 0; c < np; ++c) sum += __ldcg(sp + (size_t)c * a.P.cap);
          }
          srs[t] = 1.0f / sqrtf(sum / (float)a.K + D.eps);
        }
        named_sync(1, kWEThreads);
      }
      // the tile's sums: the segments (high plus low parts) of a group added in
      // K order, then the groups.  A later part of a split K hands its groups on
      // one by one, so the order is the same whatever the split.
      constexpr bool kGrp = w_grouped(KIND);
      const int id = rt * a.ntt + w.tt, nslot = w_slots(a.ngrp, a.nsp), later = a.ngrp / a.nsp;
      const int nc = min(TT / 2, (a.M - t0 - th * (TT / 2) + kWChunk - 1) / kWChunk * kWChunk);
      float4* part = reinterpret_cast<float4*>(a.P.part) + (size_t)id * nslot * (TT * 32) + tid;
      auto hand_on = [&](int slot, int c, const float* v) {  // columns c .. c + 3
        part[((size_t)slot * (TT / 8) + c / 4) * kWEThreads] = make_float4(v[0], v[1], v[2], v[3]);
      };
      float tot[TT / 2];
#pragma unroll
      for (int c = 0; c < TT / 2; ++c) tot[c] = 0.f;
      for (int g = w.g0; g < w.g1; ++g) {
        float acc[kGrp ? TT / 2 : 1];
        if constexpr (kGrp) {
#pragma unroll
          for (int c = 0; c < TT / 2; ++c) acc[c] = 0.f;
        }
        for (int i = 0; i < (kGrp ? a.spg : 1); ++i, ++sc) {
          if (ok) {
            ok = __all_sync(0xffffffffu, mbar_wait(&accfull[sc & 1], (uint32_t)(sc >> 1) & 1u));
            if (!ok && lane == 0) w_flag(a.B);
          }
          tc_fence_after();
          const uint32_t src =
              tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)((sc & 1) * N + th * (TT / 2));
          constexpr int kDrain = kGrp ? 8 : 16;  // (16 with two accumulators would spill)
#pragma unroll
          for (int c = 0; c < TT / 2; c += kDrain)
            if (ok && c < nc) {
              float v[kDrain];
              tc_ld_sum(src + c, src + TT + c, v);
              if constexpr (kGrp) {
#pragma unroll
                for (int j = 0; j < kDrain; ++j) acc[c + j] += v[j];
              } else if (w.sp == 0) {
#pragma unroll
                for (int j = 0; j < kDrain; ++j) tot[c + j] += v[j];
              } else {
#pragma unroll
                for (int j = 0; j < kDrain; j += 4) hand_on(g - later + 1, c + j, v + j);
              }
            }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&accempty[sc & 1]);
        }
        if constexpr (kGrp) {
#pragma unroll
          for (int c = 0; c < TT / 2; ++c) tot[c] += acc[c];
          if (w.sp > 0) {
#pragma unroll
            for (int c = 0; c < TT / 2; c += 4)
              if (c < nc) hand_on(g - later + 1, c, acc + c);
          }
        }
      }
      if (a.nsp > 1) {
        // K is split: the last block of the tile adds the partial sums in K order
        if (w.sp == 0) {
#pragma unroll
          for (int c = 0; c < TT / 2; c += 4)
            if (c < nc) hand_on(0, c, tot + c);
        }
        named_sync(1, kWEThreads);
        if (tid == 0)
          s_last = atom_add_acq_rel_gpu(a.P.tickets + id, 1u) == (uint32_t)(a.nsp - 1);
        named_sync(1, kWEThreads);
        if (!s_last) continue;
        if (tid == 0) a.P.tickets[id] = 0u;
#pragma unroll
        for (int c = 0; c < TT / 2; ++c) tot[c] = 0.f;
        for (int s = 0; s < nslot; ++s) {
          float4 u[TT / 8];  // in flight together
#pragma unroll
          for (int i = 0; i < TT / 8; ++i)
            u[i] = 4 * i < nc ? __ldcg(&part[((size_t)s * (TT / 8) + i) * kWEThreads])
                              : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int i = 0; i < TT / 8; ++i) {
            tot[4 * i] += u[i].x;
            tot[4 * i + 1] += u[i].y;
            tot[4 * i + 2] += u[i].z;
            tot[4 * i + 3] += u[i].w;
          }
        }
      }
#pragma unroll
      for (int c = 0; c < TT / 2; c += kWChunk) {
        const int tl = th * (TT / 2) + c;  // the step's first token in the tile
        if (t0 + tl >= a.M) break;
        float v[kWChunk];
#pragma unroll
        for (int j = 0; j < kWChunk; ++j) v[j] = tot[c + j];
        const int nt = min(kWChunk, a.M - t0 - tl);
        if constexpr (KIND == kWResid) {
          const int row = rt * kWR + 32 * q + lane;
          const bool in = row < a.N;
          float* h = a.P.h + (size_t)(t0 + tl) * D.d + row;
          float hp[kWChunk];
#pragma unroll
          for (int j = 0; j < kWChunk; ++j) hp[j] = (in && j < nt) ? h[(size_t)j * D.d] : 0.f;
          const float g = (in && a.gnext) ? __bfloat162float(a.gnext[row]) : 0.f;
          const size_t plane = (size_t)a.P.cap * D.d;
          __nv_bfloat16* xn = a.P.xn + (size_t)(t0 + tl) * D.d + row;
          float sq[kWChunk];
#pragma unroll
          for (int j = 0; j < kWChunk; ++j) {
            const float x = hp[j] + v[j];
            sq[j] = (in && j < nt) ? x * x : 0.f;
            if (in && j < nt) {
              h[(size_t)j * D.d] = x;
              if (a.gnext) put_split(xn + (size_t)j * D.d, plane, x * g);
            }
          }
          const float s = warp_sum16(sq, lane);
          if (!(lane & 1)) red[q * TT + tl + (lane >> 1)] = s;
        } else if constexpr (KIND == kWHead) {
          const int row = rt * kWR + 32 * q + lane;
#pragma unroll
          for (int j = 0; j < kWChunk; ++j)
            if (row < a.N && j < nt) a.B.logits[(size_t)(t0 + tl + j) * D.V + row] = v[j] * srs[tl + j];
        } else {
          // swap halves: warps of rows 0-63 finish tokens 0-7 of the step,
          // warps of rows 64-127 tokens 8-15
          const bool low = q < 2;
          float* mine = exch + ((size_t)xp * kWEpi + warp) * 256 + lane;
          const float* other = exch + ((size_t)xp * kWEpi + (warp ^ 2)) * 256 + lane;
          xp ^= 1;
#pragma unroll
          for (int j = 0; j < 8; ++j) mine[j * 32] = low ? v[8 + j] : v[j];
          named_sync(2 + th, 128);
          const int i = 32 * (q & 1) + lane;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int tj = low ? j : 8 + j;
            if (tj >= nt) continue;
            const int t = t0 + tl + tj;
            const float rs = srs[tl + tj];
            const float o = other[j * 32];
            const float y0 = (low ? v[j] : o) * rs, y1 = (low ? o : v[8 + j]) * rs;
            if constexpr (KIND == kWGateUp) {
              const int jj = rt * 64 + i;
              if (jj < D.F)
                put_split(a.P.xa + (size_t)t * D.F + jj, (size_t)a.P.cap * D.F,
                          y0 / (1.0f + expf(-y0)) * y1);
            } else {
              // one head per tile: rotary pair (i, i + 64) or two value rows
              const int head = rt, pos = a.pos0 + t;
              __nv_bfloat16* kv = static_cast<__nv_bfloat16*>(a.B.kv) +
                                  (size_t)a.layer * 2 * D.Hkv * D.max_seq * D.hd;
              if (head < D.Hq + D.Hkv) {
                const float2 cs = a.B.rope[(size_t)pos * 64 + i];
                const float r0 = y0 * cs.x - y1 * cs.y, r1 = y1 * cs.x + y0 * cs.y;
                if (head < D.Hq) {
                  float* qo = a.P.xq + (size_t)t * D.qd + head * 128 + i;
                  qo[0] = r0;
                  qo[64] = r1;
                } else {
                  __nv_bfloat16* kr = kv + ((size_t)(head - D.Hq) * D.max_seq + pos) * 128 + i;
                  kr[0] = __float2bfloat16_rn(r0);
                  kr[64] = __float2bfloat16_rn(r1);
                }
              } else {
                __nv_bfloat16* vr =
                    kv + ((size_t)(head - D.Hq) * D.max_seq + pos) * 128 + i;  // Hkv + g
                vr[0] = __float2bfloat16_rn(y0);
                vr[64] = __float2bfloat16_rn(y1);
              }
            }
          }
        }
      }
      named_sync(1, kWEThreads);
      if constexpr (KIND == kWResid) {
        for (int t = tid; t < TT && t0 + t < a.M; t += kWEThreads)
          a.ss_out[(size_t)rt * a.P.cap + t0 + t] =
              red[t] + red[TT + t] + red[2 * TT + t] + red[3 * TT + t];
        named_sync(1, kWEThreads);
      }
    }
  }
  // TMEM is released once every accumulator has been read
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kWMmaWarp) tc_dealloc(tmem, S::kCols);
}

// ------------------------------------------------------------- attention

namespace {

constexpr int kAQ = 64;   // query rows per block (16 per warp)
constexpr int kAKB = 64;  // keys per step
constexpr int kAHd = 128;
constexpr int kAWThreads = 128;
constexpr size_t kAQBytes = (size_t)3 * kAQ * kAHd * 2;  // queries, three bf16 parts
constexpr size_t kAKBytes = (size_t)kAKB * kAHd * 2;
constexpr size_t kAWSmem = kAQBytes + 4 * kAKBytes;      // + keys and values, double buffered

}  // namespace

__global__ void __launch_bounds__(kAWThreads, 2)
    k_attn_wide(const Dims D, const Bufs B, const WideBufs P, int layer, int M, int pos0) {
  extern __shared__ __align__(1024) unsigned char smem[];
  pdl_wait();
  pdl_launch_dependents();
  const int head = blockIdx.x;
  const int q0 = (int)(gridDim.y - 1 - blockIdx.y) * kAQ;  // longest blocks first
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  const int g = head / (D.Hq / D.Hkv);
  const __nv_bfloat16* kv =
      static_cast<const __nv_bfloat16*>(B.kv) + (size_t)layer * 2 * D.Hkv * D.max_seq * kAHd;
  const __nv_bfloat16* kb = kv + (size_t)g * D.max_seq * kAHd;
  const __nv_bfloat16* vb = kv + (size_t)(D.Hkv + g) * D.max_seq * kAHd;
  const uint32_t sq = smem_u32(smem), sk = sq + (uint32_t)kAQBytes;
  const int last = pos0 + min(M, q0 + kAQ) - 1;  // last key any row of the block sees
  const int nkb = last / kAKB + 1;

  auto stage = [&](int b) {
    const uint32_t kd = sk + (uint32_t)((b & 1) * 2) * (uint32_t)kAKBytes;
    const uint32_t vd = kd + (uint32_t)kAKBytes;
#pragma unroll
    for (int j = 0; j < kAKB * 16 / kAWThreads; ++j) {
      const int c = tid + j * kAWThreads, row = c >> 4, ch = c & 15;
      const int key = b * kAKB + row;
      const bool in = key <= last;  // keys past the last one read zeros
      const size_t off = (size_t)(in ? key : 0) * kAHd + ch * 8;
      cp_async16(kd + sw256(row, ch), kb + off, in);
      cp_async16(vd + sw256(row, ch), vb + off, in);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  stage(0);
  // queries: three bf16 parts
  for (int c = tid; c < kAQ * 16; c += kAWThreads) {
    const int row = c >> 4, ch = c & 15;
    float4 x0 = make_float4(0.f, 0.f, 0.f, 0.f), x1 = x0;
    if (q0 + row < M) {
      const float4* p =
          reinterpret_cast<const float4*>(P.xq + (size_t)(q0 + row) * D.qd + head * kAHd + ch * 8);
      x0 = p[0];
      x1 = p[1];
    }
    uint4 w[3];
    split3(x0.x, x0.y, w[0].x, w[1].x, w[2].x);
    split3(x0.z, x0.w, w[0].y, w[1].y, w[2].y);
    split3(x1.x, x1.y, w[0].z, w[1].z, w[2].z);
    split3(x1.z, x1.w, w[0].w, w[1].w, w[2].w);
#pragma unroll
    for (int s = 0; s < 3; ++s)
      *reinterpret_cast<uint4*>(smem + (size_t)s * kAQ * 256 + sw256(row, ch)) = w[s];
  }

  float o[16][4];
#pragma unroll
  for (int n = 0; n < 16; ++n)
#pragma unroll
    for (int e = 0; e < 4; ++e) o[n][e] = 0.f;
  float mx[2] = {-INFINITY, -INFINITY}, ls[2] = {0.f, 0.f};
  const float scale = 1.0f / sqrtf((float)kAHd);
  const int r0 = pos0 + q0 + 16 * warp + (lane >> 2);  // position of the thread's first row
  const int lrow = 16 * warp + (lane & 15), lch = lane >> 4;  // ldmatrix row / chunk of queries

  for (int b = 0; b < nkb; ++b) {
    if (b + 1 < nkb) {
      stage(b + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const uint32_t kd = sk + (uint32_t)((b & 1) * 2) * (uint32_t)kAKBytes;
    const uint32_t vd = kd + (uint32_t)kAKBytes;
    float s[8][4];
#pragma unroll
    for (int n = 0; n < 8; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) s[n][e] = 0.f;
    // the queries' two lower parts first: the running sum is cut at its own
    // last place, so the small terms lose nothing to it
#pragma unroll
    for (int pass = 0; pass < 2; ++pass)
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        uint32_t qa[2][4];
        const int np = pass ? 1 : 2;
#pragma unroll
        for (int p = 0; p < np; ++p)
          ldsm4(sq + (uint32_t)((pass ? 0 : 2 - p) * kAQ * 256) + sw256(lrow, 2 * kk + lch), qa[p]);
        // keys 16 n2 .. + 15 x 16 columns: two n-tiles
        uint32_t kf[4][4];
#pragma unroll
        for (int n2 = 0; n2 < 4; ++n2)
          ldsm4(kd + sw256(16 * n2 + (lane & 7) + ((lane >> 4) << 3), 2 * kk + ((lane >> 3) & 1)),
                kf[n2]);
#pragma unroll
        for (int p = 0; p < np; ++p)
#pragma unroll
          for (int n2 = 0; n2 < 4; ++n2) {
            mma16816(s[2 * n2], qa[p], kf[n2][0], kf[n2][1]);
            mma16816(s[2 * n2 + 1], qa[p], kf[n2][2], kf[n2][3]);
          }
      }
    // scale, causal mask, running maximum
    const int kbase = b * kAKB + 2 * (lane & 3);
    float nm[2] = {mx[0], mx[1]};
#pragma unroll
    for (int n = 0; n < 8; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int key = kbase + 8 * n + (e & 1), row = r0 + 8 * (e >> 1);
        s[n][e] = key <= row ? s[n][e] * scale : -INFINITY;
        nm[e >> 1] = fmaxf(nm[e >> 1], s[n][e]);
      }
    float f[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      nm[r] = fmaxf(nm[r], __shfl_xor_sync(0xffffffffu, nm[r], 1));
      nm[r] = fmaxf(nm[r], __shfl_xor_sync(0xffffffffu, nm[r], 2));
      // block 0 holds key 0, which every row sees: the maximum is finite
      f[r] = expf(mx[r] - nm[r]);
      mx[r] = nm[r];
      ls[r] *= f[r];
    }
#pragma unroll
    for (int n = 0; n < 8; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        s[n][e] = expf(s[n][e] - mx[e >> 1]);
        ls[e >> 1] += s[n][e];
      }
    uint32_t pa[4][3][4];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        split3(s[2 * ks + (e >> 1)][2 * (e & 1)], s[2 * ks + (e >> 1)][2 * (e & 1) + 1],
               pa[ks][0][e], pa[ks][1][e], pa[ks][2][e]);
#pragma unroll
    for (int n4 = 0; n4 < 4; ++n4) {
      // this step's share of 32 columns in sums of its own (four chains, to
      // cover the latency of mma.sync), then one rounded fused multiply-add
      // into the running output
      float t[4][4];
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) t[n][e] = 0.f;
      uint32_t vf[2][4][4];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
          ldsm4t(vd + sw256(16 * ks + (lane & 15), 4 * n4 + 2 * h + (lane >> 4)), vf[h][ks]);
#pragma unroll
      for (int p = 2; p >= 0; --p)
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            mma16816(t[2 * h], pa[ks][p], vf[h][ks][0], vf[h][ks][1]);
            mma16816(t[2 * h + 1], pa[ks][p], vf[h][ks][2], vf[h][ks][3]);
          }
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[4 * n4 + n][e] = fmaf(o[4 * n4 + n][e], f[e >> 1], t[n][e]);
    }
    __syncthreads();  // the buffer is staged again two steps on
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    ls[r] += __shfl_xor_sync(0xffffffffu, ls[r], 1);
    ls[r] += __shfl_xor_sync(0xffffffffu, ls[r], 2);
  }
  const size_t plane = (size_t)P.cap * D.qd;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int m = q0 + 16 * warp + (lane >> 2) + 8 * r;
    if (m >= M) continue;
    __nv_bfloat16* out = P.xo + (size_t)m * D.qd + head * kAHd + 2 * (lane & 3);
#pragma unroll
    for (int n = 0; n < 16; ++n) {
      const float x = o[n][2 * r] / ls[r], y = o[n][2 * r + 1] / ls[r];
      const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
      const __nv_bfloat162 l =
          __floats2bfloat162_rn(x - __low2float(h), y - __high2float(h));
      *reinterpret_cast<__nv_bfloat162*>(out + 8 * n) = h;
      *reinterpret_cast<__nv_bfloat162*>(out + plane + 8 * n) = l;
    }
  }
}

// ------------------------------------------------------------- embedding

// Row m of a chunk: h = embed[tok[m]], its split parts under the first norm's
// weights, and its sums of squares per 128 columns.
__global__ void __launch_bounds__(256)
    k_embed_wide(const Dims D, const Bufs B, const WideBufs P, const __nv_bfloat16* __restrict__ emb,
                 const __nv_bfloat16* __restrict__ gnorm, const int32_t* __restrict__ toks) {
  pdl_wait();
  pdl_launch_dependents();
  const int m = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int tok = toks[m];
  if (tok < 0 || tok >= D.V) {
    if (threadIdx.x == 0) atomicOr(&B.ctl->err, (int)kErrToken);
    tok = 0;
  }
  const __nv_bfloat16* row = emb + (size_t)tok * D.d;
  float* h = P.h + (size_t)m * D.d;
  __nv_bfloat16* xn = P.xn + (size_t)m * D.d;
  const size_t plane = (size_t)P.cap * D.d;
  for (int c = warp; c * kWR < D.d; c += 8) {
    float sp = 0.f;
#pragma unroll
    for (int j = 0; j < kWR / 32; ++j) {
      const int i = c * kWR + j * 32 + lane;
      if (i < D.d) {
        const float v = __bfloat162float(row[i]);
        h[i] = v;
        put_split(xn + i, plane, v * __bfloat162float(gnorm[i]));
        sp = fmaf(v, v, sp);
      }
    }
    sp = warp_sum(sp);
    if (lane == 0) P.ss[(size_t)c * P.cap + m] = sp;
  }
}

// ------------------------------------------------------------- host side

namespace {

template <int TT, int KIND>
cudaError_t wide_prep() {
  return cudaFuncSetAttribute(k_wide<TT, KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)WL<TT>::total);
}
template <int TT>
cudaError_t wide_prep_all() {
  cudaError_t e = wide_prep<TT, kWQkv>();
  if (e == cudaSuccess) e = wide_prep<TT, kWResid>();
  if (e == cudaSuccess) e = wide_prep<TT, kWHead>();
  return e != cudaSuccess ? e : wide_prep<TT, kWGateUp>();
}

// Cycles of one 64-column stage of a tile of tt tokens on one SM: the copy of
// its 16 KB of weights and 256 tt bytes of input rows out of L2 (about 60
// bytes a cycle and SM with all SMs reading), or 4 tt cycles of tcgen05.mma.
int stage_cost(int tt) { return 273 + 4 * tt + tt / 4; }

int row_tiles(int N, bool pairs) { return pairs ? (N / 2 + 63) / 64 : (N + kWR - 1) / kWR; }

// How K is cut, by the matrix and the device alone: into as many equal groups as
// one token tile's row tiles leave SMs for (at most eight, none shorter than
// kWSeg stages), which are the parts of a short prompt, and a group into as few
// segments as kWSeg allows.  Where segments are not added in groups each is a
// group of its own.
struct KCut {
  int ngrp, spg;
};
KCut cut_k(int sms, int nrt, int nks, bool grouped) {
  const int groups = std::max(1, std::min({8, sms / nrt, nks / kWSeg}));
  const int spg = (nks + groups * kWSeg - 1) / (groups * kWSeg);
  return grouped ? KCut{groups, spg} : KCut{groups * spg, 1};
}

// Token tile (index 0, 1, 2 = 32, 64, 128 tokens) and parts of K of the product
// of nrt row tiles x nks stages with M tokens that have the least work on the
// busiest SM.  K is split only where that still leaves every block its own
// SM; the join costs about 6000 cycles (the parts' stores, the ticket's round
// trip) and the parts' way back through L2.
struct WPlan {
  int ti, nsp;
  long long cost;
};
WPlan pick_plan(int sms, int nrt, int nks, int M, bool grouped) {
  WPlan best{0, 1, -1};
  const int groups = cut_k(sms, nrt, nks, grouped).ngrp;
  for (int i = 0; i < 3; ++i) {
    const int tt = 32 << i;
    const long long tiles = (long long)nrt * ((M + tt - 1) / tt);
    for (int nsp = 1; nsp <= 8; ++nsp) {
      if (nsp > 1 && (nsp > groups || tiles * nsp > sms ||
                      tiles * w_slots(groups, nsp) * tt > (long long)kWideParts * 128))
        break;
      const int most = ((groups + nsp - 1) / nsp * nks + groups - 1) / groups;
      const long long c = (tiles * nsp + sms - 1) / sms * most * stage_cost(tt) +
                          (nsp > 1 ? 6000 + 9LL * w_slots(groups, nsp) * tt : 0);
      if (best.cost < 0 || c < best.cost) best = WPlan{i, nsp, c};
    }
  }
  return best;
}

template <int KIND>
cudaError_t wide_launch(const CUtensorMap& wm, const CUtensorMap* xm, WArgs& a, cudaStream_t st) {
  a.nks = (a.K + kWK - 1) / kWK;
  a.nrt = row_tiles(a.N, KIND == kWGateUp);
  const WPlan p = pick_plan(a.D.num_sms, a.nrt, a.nks, a.M, w_grouped(KIND));
  const KCut cut = cut_k(a.D.num_sms, a.nrt, a.nks, w_grouped(KIND));
  a.ntt = (a.M + (32 << p.ti) - 1) / (32 << p.ti);
  a.ngrp = cut.ngrp;
  a.spg = cut.spg;
  a.seg_q = a.nks / (a.ngrp * a.spg);
  a.seg_r = a.nks % (a.ngrp * a.spg);
  a.nsp = p.nsp;
  const long long tiles = (long long)a.nrt * a.ntt * a.nsp;
  const dim3 grid((unsigned)(tiles < a.D.num_sms ? tiles : a.D.num_sms)), blk(kWThreads);
  switch (p.ti) {
    case 0: return launch_ex(k_wide<32, KIND>, grid, blk, WL<32>::total, st, wm, xm[0], a);
    case 1: return launch_ex(k_wide<64, KIND>, grid, blk, WL<64>::total, st, wm, xm[1], a);
    default: return launch_ex(k_wide<128, KIND>, grid, blk, WL<128>::total, st, wm, xm[2], a);
  }
}

}  // namespace

bool encode_wide_maps(CUtensorMap (&m)[3], const void* x, int cols, int cap) {
  for (int i = 0; i < 3; ++i)
    if (!encode_split_map(&m[i], x, cols, cap, 32 << i)) return false;
  return true;
}

cudaError_t prepare_wide_kernels() {
  cudaError_t e;
  if ((e = wide_prep_all<32>()) != cudaSuccess) return e;
  if ((e = wide_prep_all<64>()) != cudaSuccess) return e;
  if ((e = wide_prep_all<128>()) != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_attn_wide, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kAWSmem);
}

// Work of one layer of a chunk of M rows on the busiest SM (stage cycles).
long long wide_layer_cost(const Dims& D, int M) {
  auto mat = [&](int kind, int N, int K) {
    return pick_plan(D.num_sms, row_tiles(N, kind == kWGateUp), (K + kWK - 1) / kWK, M, w_grouped(kind)).cost;
  };
  return mat(kWQkv, (D.Hq + 2 * D.Hkv) * D.hd, D.d) + mat(kWResid, D.d, D.qd) +
         mat(kWGateUp, 2 * D.F, D.d) + mat(kWResid, D.d, D.F);
}

cudaError_t launch_embed_wide(const Dims& D, const Bufs& B, const WideBufs& P, const void* embed,
                              const void* gnorm, const int32_t* toks, int M, cudaStream_t st) {
  return launch_ex(k_embed_wide, dim3(M), dim3(256), 0, st, D, B, P,
                   static_cast<const __nv_bfloat16*>(embed),
                   static_cast<const __nv_bfloat16*>(gnorm), toks);
}

cudaError_t launch_head_wide(const Dims& D, const Bufs& B, const WideBufs& P, const WideMaps& xm,
                             const CUtensorMap& lm, int row0, int M, cudaStream_t st) {
  WArgs a{};
  a.D = D;
  a.B = B;
  a.P = P;
  a.M = M;
  a.row0 = row0;
  a.N = D.V;
  a.K = D.d;
  a.ss_in = P.ss + row0;  // written by the last layer's down projection
  return wide_launch<kWHead>(lm, xm.xn, a, st);
}

cudaError_t launch_layer_wide(const Dims& D, const Bufs& B, const WideBufs& P, const WideMaps& xm,
                              const LayerW& w, const void* next_norm, int layer, int M, int pos0,
                              cudaStream_t st) {
  float* ss[2] = {P.ss, P.ss + (size_t)((D.d + kWR - 1) / kWR) * P.cap};
  WArgs a{};
  a.D = D;
  a.B = B;
  a.P = P;
  a.M = M;
  a.pos0 = pos0;
  a.layer = layer;
  cudaError_t e;
  // RMSNorm + QKV + RoPE + KV rows
  a.N = (D.Hq + 2 * D.Hkv) * D.hd;
  a.K = D.d;
  a.ss_in = ss[0];
  if ((e = wide_launch<kWQkv>(*w.tm[0], xm.xn, a, st)) != cudaSuccess) return e;
  if ((e = launch_ex(k_attn_wide, dim3(D.Hq, (M + kAQ - 1) / kAQ), dim3(kAWThreads), kAWSmem, st, D,
                     B, P, layer, M, pos0)) != cudaSuccess)
    return e;
  // O projection + residual
  a.N = D.d;
  a.K = D.qd;
  a.ss_in = nullptr;
  a.ss_out = ss[1];
  a.gnext = static_cast<const __nv_bfloat16*>(w.ffn_norm);
  if ((e = wide_launch<kWResid>(*w.tm[1], xm.xo, a, st)) != cudaSuccess) return e;
  // RMSNorm + gate/up + SwiGLU
  a.N = 2 * D.F;
  a.K = D.d;
  a.ss_in = ss[1];
  if ((e = wide_launch<kWGateUp>(*w.tm[2], xm.xn, a, st)) != cudaSuccess) return e;
  // down projection + residual
  a.N = D.d;
  a.K = D.F;
  a.ss_in = nullptr;
  a.ss_out = ss[0];
  a.gnext = static_cast<const __nv_bfloat16*>(next_norm);
  return wide_launch<kWResid>(*w.tm[3], xm.xa, a, st);
}

}  // namespace ssd
