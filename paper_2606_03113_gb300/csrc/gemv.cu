// gemv.cu -- the weight-streaming matrix-vector product of the kernel-level
// entry points: ssd_op_gemv of fp32 models and ssd_gemv_noalloc.  (A model's
// own passes run on fp32.cu, fp32, and tile.cu and wide.cu, bf16.)
//
// y[m] = W x[m] for M <= 17 fp32 input rows, one persistent grid of one block
// per SM:
//  - the matrix is cut into units of 32 rows x 512 bytes; the units, in
//    (row tile, K) order, are split evenly over the blocks ("stream-K"), so
//    every SM streams the same number of bytes whatever the matrix shape, and
//    a block copies up to four consecutive units of a tile as one stage;
//  - a producer warp copies each stage into a 3-deep shared-memory ring with
//    1-D bulk async copies (one copy of up to 2 KB per row: smaller copies
//    starve the copy engine; evict-first in L2), synchronised by
//    mbarriers; its copies do not wait for the previous kernel (programmatic
//    dependent launch);
//  - eight consumer warps read the stage from shared memory (four rows per
//    warp, so each input load serves four rows; 16 bytes per lane per
//    512-byte step), multiply with the fp32 input rows (from L1/L2) and
//    accumulate; a 32-row tile is reduced with warp shuffles;
//  - a tile split between two blocks is finished by whichever block completes
//    its share last (per-tile ticket), which adds the partial sums in block
//    order, so results do not depend on scheduling.
#include <math.h>

#include <mutex>
#include <type_traits>

#include "kernels.h"
#include "pipe.cuh"

namespace ssd {

constexpr int kRT = 32;             // rows per tile
constexpr int kRowBytes = 2048;     // bytes of one row per stage (4 units)
constexpr int kUnit = 512;          // bytes of one row per assignment unit
constexpr int kNS = 3;              // ring depth
constexpr int kCWarps = 8;          // consumer warps
constexpr int kCThreads = kCWarps * 32;
constexpr int kThreads = kCThreads + 32;  // + producer warp
constexpr int kRowStride = kRowBytes + 16;  // padded row pitch in shared memory:
                                            // rows of an 8x8 ldmatrix land on distinct banks
constexpr int kStageBytes = kRT * kRowStride;
constexpr int kNB = (kMaxM + 7) / 8;        // 8-token column blocks of the tensor-core path

struct Geom {
  int N, K;          // rows, columns (elements)
  int nks;           // 512-byte units per row (per tile)
  int ntiles;
  long long T;       // units (tiles x nks)
  int P;             // blocks
  int row_bytes;     // K * elt
  int elt;           // element size in bytes
};

struct StreamArgs {
  Geom g;
  Dims D;
  Bufs B;
  const void* W;
  const float* x;        // [M][K] fp32 input rows
  float* y;              // [M][N] products
  int M;
};

__host__ __device__ inline long long stage_start(const Geom& g, int b) {
  return g.T * (long long)b / g.P;
}

__device__ inline int block_of_stage(const Geom& g, long long s) {
  int b = (int)(s * g.P / g.T);
  if (b >= g.P) b = g.P - 1;
  while (b + 1 < g.P && stage_start(g, b + 1) <= s) ++b;
  while (b > 0 && stage_start(g, b) > s) --b;
  return b;
}

// Global row of local row r (0..31) of a tile, or -1 past the end.  Consumer
// warp w handles the local rows w, w + 8, w + 16 and w + 24.
__device__ inline int map_row(const Geom& g, int tile, int r) {
  const int row = tile * kRT + r;
  return row < g.N ? row : -1;
}

struct SmemLayout {
  static constexpr size_t ring = 0;
  static constexpr size_t bars = ring + (size_t)kNS * kStageBytes;
  static constexpr size_t flag = bars + 2 * kNS * sizeof(uint64_t);
  static constexpr size_t red = flag + 64;
  template <int MM>
  static constexpr size_t total() {  // + tensor-core partial sums [4 K-quarters][32][8 kNB]
    return red + sizeof(float) * 4 * kRT * 8 * kNB;
  }
};

// ------------------------------------------------------------ the kernel

template <int MM>
__device__ __forceinline__ float pick(const float (&v)[MM], int lane) {
  float r = 0.f;
#pragma unroll
  for (int m = 0; m < MM; ++m)
    if (m == lane) r = v[m];
  return r;
}

// ---- tensor-core helpers (verification rows: M > 1)
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& a0, uint32_t& a1, uint32_t& a2,
                                        uint32_t& a3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(a0), "=r"(a1), "=r"(a2), "=r"(a3)
               : "r"(addr));
}

// d += A(16x16, bf16, row) * B(16x8, bf16, col), fp32 accumulate.
__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                          uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Splits (x0, x1) into bf16 high parts and bf16 residuals, packed low-k first:
// x = hi + lo to about 16 significant bits, so two bf16 products keep the
// activations' fp32 precision.
__device__ __forceinline__ void split_bf16x2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat16 h0 = __float2bfloat16_rn(x0), h1 = __float2bfloat16_rn(x1);
  const __nv_bfloat16 l0 = __float2bfloat16_rn(x0 - __bfloat162float(h0));
  const __nv_bfloat16 l1 = __float2bfloat16_rn(x1 - __bfloat162float(h1));
  hi = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
  lo = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
}

// Stage sequence of a block: from unit u, the run of up to 4 units that stays
// inside the tile and the block's range.  Producer and consumers walk it
// identically.
__device__ __forceinline__ int stage_units(const Geom& g, long long u, long long u_end) {
  const long long j = u % g.nks;
  long long n = g.nks - j;
  if (n > kRowBytes / kUnit) n = kRowBytes / kUnit;
  if (n > u_end - u) n = u_end - u;
  return (int)n;
}

template <typename T, int MM, bool MMA>
__global__ void __launch_bounds__(kThreads, 1) k_stream(const StreamArgs a) {
  static_assert(!MMA || (std::is_same<T, __nv_bfloat16>::value && MM > 1), "tensor path: bf16 rows");
  extern __shared__ __align__(128) unsigned char smem[];
  using E = Elem<T>;
  constexpr int EPC = E::kPerChunk;
  constexpr int CU = kUnit / (int)sizeof(T);  // columns per unit
  unsigned char* ring = smem + SmemLayout::ring;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + SmemLayout::bars);
  uint64_t* empty = full + kNS;
  int* flag = reinterpret_cast<int*>(smem + SmemLayout::flag);

  const Geom& g = a.g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long u_begin = stage_start(g, blockIdx.x), u_end = stage_start(g, blockIdx.x + 1);
  if (threadIdx.x == 0) {
    for (int i = 0; i < kNS; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kCWarps);
    }
    mbar_init_fence();
  }
  __syncthreads();
  pdl_launch_dependents();

  if (warp == kCWarps) {
    // ---------------- producer: weights do not depend on earlier kernels
    const unsigned char* W = static_cast<const unsigned char*>(a.W);
    const uint64_t pol = evict_first_policy();
    int i = 0;
    for (long long u = u_begin; u < u_end; ++i) {
      const int n = stage_units(g, u, u_end);
      const int slot = i % kNS;
      const uint32_t ph = (uint32_t)(i / kNS) & 1u;
      if (!mbar_wait(&empty[slot], ph ^ 1u)) {
        if (lane == 0) atomicOr(&a.B.ctl->err, (int)kErrTimeout);
        break;
      }
      const int tile = (int)(u / g.nks), j = (int)(u - (long long)tile * g.nks);
      const int off = j * kUnit;
      const int bytes = min(n * kUnit, g.row_bytes - off);
      const int row = map_row(g, tile, lane);
      const int nvalid = __popc(__ballot_sync(0xffffffffu, row >= 0));
      if (lane == 0) mbar_arrive_expect_tx(&full[slot], (uint32_t)(nvalid * bytes));
      __syncwarp();
      if (row >= 0)
        bulk_g2s(ring + (size_t)slot * kStageBytes + lane * kRowStride,
                 W + (size_t)row * g.row_bytes + off, (uint32_t)bytes, &full[slot], pol);
      u += n;
    }
    // drain: the copies of the last stages have landed before the block exits
    if (lane == 0)
      for (int k = i > kNS ? i - kNS : 0; k < i; ++k) mbar_wait(&full[k % kNS], (uint32_t)(k / kNS) & 1u);
    return;
  }

  // ---------------- consumers
  pdl_wait();
  const int M = a.M;
  const int tid = threadIdx.x;
  const float* x = a.x;
  float acc[MMA ? 1 : 4][MMA ? 1 : MM];
  float dmm[kNB][4];  // tensor-core accumulators: rows rb*16 + (g, g+8), tokens nb*8 + 2c + (0, 1)
  float* red = reinterpret_cast<float*>(smem + SmemLayout::red);
  const int rloc[4] = {warp, warp + 8, warp + 16, warp + 24};
  // lane m holds input row m's products with the warp's four rows
  auto store = [&](int tile, const float (&v)[4]) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int row = map_row(g, tile, rloc[r]);
      if (lane < M && row >= 0) a.y[(size_t)lane * g.N + row] = v[r];
    }
  };
  int cur = -1;
  bool ok = true;
  int i = 0;
  for (long long u = u_begin; u < u_end; ++i) {
    const int n = stage_units(g, u, u_end);
    const int slot = i % kNS;
    const uint32_t ph = (uint32_t)(i / kNS) & 1u;
    const int tile = (int)(u / g.nks), j = (int)(u - (long long)tile * g.nks);
    u += n;
    if (tile != cur) {
      if (MMA) {
#pragma unroll
        for (int nb = 0; nb < kNB; ++nb)
#pragma unroll
          for (int q = 0; q < 4; ++q) dmm[nb][q] = 0.f;
      } else {
#pragma unroll
        for (int r = 0; r < (MMA ? 1 : 4); ++r)
#pragma unroll
          for (int m = 0; m < (MMA ? 1 : MM); ++m) acc[r][m] = 0.f;
      }
      cur = tile;
    }
    if (ok && !mbar_wait(&full[slot], ph)) {
      if (lane == 0) atomicOr(&a.B.ctl->err, (int)kErrTimeout);
      ok = false;
    }
    const int bytes = min(n * kUnit, g.row_bytes - j * kUnit);
    const unsigned char* stg = ring + (size_t)slot * kStageBytes + lane * 16;
    const int col0 = j * CU + lane * 16 / (int)sizeof(T);
    if constexpr (MMA) {
      // warp = (16-row block rb, 512-byte unit kq of the stage)
      const int rb = warp & 1, kq = warp >> 1;
      if (ok && kq < n) {
        const int ub = min(kUnit, bytes - kq * kUnit);
        const uint32_t abase =
            smem_u32(ring + (size_t)slot * kStageBytes + (rb * 16 + (lane & 15)) * kRowStride +
                     kq * kUnit + (lane >> 4) * 16);
        const int kc0 = (j + kq) * CU + 2 * (lane & 3);
        const int tok0 = lane >> 2;
        for (int kk = 0; kk < ub / 32; ++kk) {
          uint32_t a0, a1, a2, a3;
          ldsm_x4(abase + kk * 32, a0, a1, a2, a3);
          const int kc = kc0 + kk * 16;
#pragma unroll
          for (int nb = 0; nb < kNB; ++nb) {
            if (nb * 8 < M) {
              const int tok = nb * 8 + tok0;
              float2 xa = make_float2(0.f, 0.f), xb = make_float2(0.f, 0.f);
              if (tok < M) {
                xa = __ldg(reinterpret_cast<const float2*>(x + (size_t)tok * g.K + kc));
                xb = __ldg(reinterpret_cast<const float2*>(x + (size_t)tok * g.K + kc + 8));
              }
              uint32_t h0, l0, h1, l1;
              split_bf16x2(xa.x, xa.y, h0, l0);
              split_bf16x2(xb.x, xb.y, h1, l1);
              mma_16816(dmm[nb], a0, a1, a2, a3, h0, h1);
              mma_16816(dmm[nb], a0, a1, a2, a3, l0, l1);
            }
          }
        }
      }
    } else if (ok && bytes == kRowBytes) {
      // full stage; the single-row kernel issues every load of the stage
      // before the math, the multi-row one goes one 512-byte step at a time
      constexpr int NSUB = kRowBytes / kUnit;
      constexpr int HOIST = MM <= 2 ? NSUB : 1;
#pragma unroll
      for (int sg = 0; sg < NSUB; sg += HOIST) {
        uint4 wq[HOIST][4];
#pragma unroll
        for (int h = 0; h < HOIST; ++h)
#pragma unroll
          for (int r = 0; r < 4; ++r)
            wq[h][r] = *reinterpret_cast<const uint4*>(stg + rloc[r] * kRowStride + (sg + h) * kUnit);
#pragma unroll
        for (int m = 0; m < MM; ++m) {
          if (m < M) {
            float4 xq[HOIST][EPC / 4];
#pragma unroll
            for (int h = 0; h < HOIST; ++h)
#pragma unroll
              for (int q = 0; q < EPC / 4; ++q)
                xq[h][q] = __ldg(reinterpret_cast<const float4*>(x + (size_t)m * g.K + col0 +
                                                                 (sg + h) * CU) + q);
#pragma unroll
            for (int h = 0; h < HOIST; ++h) {
              float xv[EPC];
#pragma unroll
              for (int q = 0; q < EPC / 4; ++q) {
                xv[4 * q] = xq[h][q].x;
                xv[4 * q + 1] = xq[h][q].y;
                xv[4 * q + 2] = xq[h][q].z;
                xv[4 * q + 3] = xq[h][q].w;
              }
#pragma unroll
              for (int r = 0; r < 4; ++r) {
                float wf[EPC];
                E::unpack(wq[h][r], wf);
#pragma unroll
                for (int e = 0; e < EPC; ++e) acc[r][m] = fmaf(wf[e], xv[e], acc[r][m]);
              }
            }
          }
        }
      }
    } else if (ok) {
      // partial stage (block range edge or ragged end of the row)
      for (int off = lane * 16; off < bytes; off += kUnit) {
        const int col = j * CU + off / (int)sizeof(T);
        float wf[4][EPC];
#pragma unroll
        for (int r = 0; r < 4; ++r)
          E::unpack(*reinterpret_cast<const uint4*>(ring + (size_t)slot * kStageBytes +
                                                    rloc[r] * kRowStride + off), wf[r]);
#pragma unroll
        for (int m = 0; m < MM; ++m) {
          if (m < M) {
            float xv[EPC];
            const float4* xp = reinterpret_cast<const float4*>(x + (size_t)m * g.K + col);
#pragma unroll
            for (int q = 0; q < EPC / 4; ++q) {
              const float4 t4 = __ldg(xp + q);
              xv[4 * q] = t4.x;
              xv[4 * q + 1] = t4.y;
              xv[4 * q + 2] = t4.z;
              xv[4 * q + 3] = t4.w;
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
              for (int e = 0; e < EPC; ++e) acc[r][m] = fmaf(wf[r][e], xv[e], acc[r][m]);
          }
        }
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[slot]);
    if (j + n != g.nks && u != u_end) continue;

    // ---- tile flush: warp-local unless the tile is shared with other blocks
    float val[4];  // lane m: the four rows' sums for input row m
    if constexpr (MMA) {
      // four K-quarter partials per row, added in quarter order
      named_sync(1, kCThreads);
      const int rb = warp & 1, kq = warp >> 1, gq = lane >> 2, cq = lane & 3;
#pragma unroll
      for (int nb = 0; nb < kNB; ++nb)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int row = rb * 16 + gq + (q >> 1) * 8, tok = nb * 8 + 2 * cq + (q & 1);
          red[((kq * kRT) + row) * 8 * kNB + tok] = dmm[nb][q];
        }
      named_sync(1, kCThreads);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float t = 0.f;
        if (lane < M)
          for (int q = 0; q < 4; ++q) t += red[((q * kRT) + rloc[r]) * 8 * kNB + lane];
        val[r] = t;
      }
    } else {
#pragma unroll
      for (int r = 0; r < (MMA ? 1 : 4); ++r)
#pragma unroll
        for (int m = 0; m < (MMA ? 1 : MM); ++m)
          if (m < M) acc[r][m] = warp_sum(acc[r][m]);
#pragma unroll
      for (int r = 0; r < (MMA ? 1 : 4); ++r) val[r] = pick(acc[r], lane);
    }
    const long long t0 = (long long)tile * g.nks, t1 = t0 + g.nks;
    if (t0 >= u_begin && t1 <= u_end) {
      store(tile, val);
      continue;
    }
    // shared with neighbouring blocks: publish this block's partial sums
    const int first_tile = (int)(u_begin / g.nks);
    const int slot2 = tile == first_tile ? 0 : 1;
    float* mine = a.B.gpart + ((size_t)blockIdx.x * 2 + slot2) * kRT * kMaxM;
    if (lane < M)
#pragma unroll
      for (int r = 0; r < 4; ++r) mine[rloc[r] * kMaxM + lane] = val[r];
    __threadfence();
    named_sync(1, kCThreads);
    const int b0 = block_of_stage(g, t0), b1 = block_of_stage(g, t1 - 1);
    if (tid == 0) {
      int contrib = 0;
      for (int b = b0; b <= b1; ++b) contrib += stage_start(g, b) < stage_start(g, b + 1);
      *flag = atomicAdd(&a.B.tile_counter[tile], 1u) == (unsigned)(contrib - 1);
    }
    named_sync(1, kCThreads);
    if (!*flag) continue;
    __threadfence();
    float uu[4] = {0.f, 0.f, 0.f, 0.f};
    if (lane < M)
      for (int b = b0; b <= b1; ++b) {  // block order: independent of who finishes
        const long long sb = stage_start(g, b);
        if (sb == stage_start(g, b + 1)) continue;
        const int sl = tile == (int)(sb / g.nks) ? 0 : 1;
        const float* p = a.B.gpart + ((size_t)b * 2 + sl) * kRT * kMaxM;
#pragma unroll
        for (int r = 0; r < 4; ++r) uu[r] += __ldcg(&p[rloc[r] * kMaxM + lane]);
      }
    if (tid == 0) a.B.tile_counter[tile] = 0u;
    store(tile, uu);
  }
}

// ------------------------------------------------------------- launchers

bool g_pdl_enabled = true;
bool g_chain_enabled = true;
thread_local bool g_pdl_ok = true;

static Geom make_geom(const Dims& D, int N, int K, int elt) {
  Geom g{};
  g.N = N;
  g.K = K;
  g.elt = elt;
  g.row_bytes = K * elt;
  g.nks = (g.row_bytes + kUnit - 1) / kUnit;
  g.ntiles = (N + kRT - 1) / kRT;
  g.T = (long long)g.ntiles * g.nks;
  g.P = D.num_sms;
  return g;
}

// Multi-row bf16 matrices whose rows are whole 512-byte units go through the
// tensor cores; single rows, fp32 and ragged rows through CUDA cores.
template <typename T, int MM>
static bool use_mma(const Geom& g) {
  return std::is_same<T, __nv_bfloat16>::value && MM > 1 && g.row_bytes % kUnit == 0;
}

template <typename T, int MM>
static cudaError_t stream_launch(const StreamArgs& a, cudaStream_t st) {
  constexpr bool kCan = std::is_same<T, __nv_bfloat16>::value && MM > 1;
  if (kCan && use_mma<T, MM>(a.g))
    return launch_ex(k_stream<T, MM, kCan>, dim3(a.g.P), dim3(kThreads), SmemLayout::total<MM>(), st,
                     a);
  return launch_ex(k_stream<T, MM, false>, dim3(a.g.P), dim3(kThreads), SmemLayout::total<MM>(), st,
                   a);
}

template <typename T, int MM>
static cudaError_t prepare_one() {
  static_assert(SmemLayout::total<MM>() <= 227 * 1024, "shared memory budget");
  constexpr bool kCan = std::is_same<T, __nv_bfloat16>::value && MM > 1;
  cudaError_t e = cudaFuncSetAttribute(k_stream<T, MM, false>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)SmemLayout::total<MM>());
  if (e != cudaSuccess || !kCan) return e;
  return cudaFuncSetAttribute(k_stream<T, MM, kCan>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)SmemLayout::total<MM>());
}

cudaError_t prepare_gemv_kernels() {
  cudaError_t e;
  if ((e = prepare_one<float, 1>()) != cudaSuccess) return e;
  if ((e = prepare_one<float, kMaxM>()) != cudaSuccess) return e;
  if ((e = prepare_one<__nv_bfloat16, 1>()) != cudaSuccess) return e;
  return prepare_one<__nv_bfloat16, kMaxM>();
}

template <typename T, int MM>
static cudaError_t plain_t(const Dims& D, const Bufs& B, const void* W, int rows, int cols,
                           const float* x, int M, float* y, cudaStream_t st) {
  StreamArgs a{};
  a.D = D;
  a.B = B;
  a.g = make_geom(D, rows, cols, (int)sizeof(T));
  a.W = W;
  a.x = x;
  a.y = y;
  a.M = M;
  return stream_launch<T, MM>(a, st);
}

cudaError_t launch_gemv_plain(const Dims& D, const Bufs& B, int dtype, const void* W, int rows,
                              int cols, const float* x, int M, float* y, cudaStream_t st) {
  if (dtype == SSD_DTYPE_BF16)
    return M == 1 ? plain_t<__nv_bfloat16, 1>(D, B, W, rows, cols, x, M, y, st)
                  : plain_t<__nv_bfloat16, kMaxM>(D, B, W, rows, cols, x, M, y, st);
  return M == 1 ? plain_t<float, 1>(D, B, W, rows, cols, x, M, y, st)
                : plain_t<float, kMaxM>(D, B, W, rows, cols, x, M, y, st);
}


// ----------------------------------------------- allocation-free variant
//
// ssd_gemv_noalloc: the plain weight-streaming product for callers that can
// not allocate device memory.  Its scratch -- the partial sums of row tiles
// shared by two blocks, their tickets and an error word -- lives in one
// file-scope device array instead of a caller-provided workspace.

constexpr int kNoAllocBlocks = 256;   // grid cap (one block per SM)
constexpr int kNoAllocTiles = 4096;   // row tiles of 32: rows <= 131072
constexpr size_t kNoAllocPart = sizeof(float) * (size_t)kNoAllocBlocks * 2 * kRT * kMaxM;
constexpr size_t kNoAllocCount = sizeof(uint32_t) * kNoAllocTiles;
constexpr size_t kNoAllocCtl = (sizeof(Ctl) + 255) / 256 * 256;
constexpr size_t kNoAllocBytes = kNoAllocPart + kNoAllocCount + kNoAllocCtl;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

namespace {
struct NoAllocDevice {
  bool ready = false;
  unsigned char* scratch = nullptr;  // device address of g_noalloc_scratch
  int sms = 0;
};
std::mutex g_noalloc_mu;
NoAllocDevice g_noalloc_dev[64];
}  // namespace

}  // namespace ssd

extern "C" ssd_status ssd_gemv_noalloc(const void* W, int32_t dtype, int32_t rows, int32_t cols,
                                       const float* x_dev, int32_t M, float* y_dev,
                                       int32_t* err_dev, void* stream) {
  using namespace ssd;
  if (!W || !x_dev || !y_dev || ((uintptr_t)W & 15u) || ((uintptr_t)x_dev & 15u))
    return SSD_ERR_INVALID_ARG;
  if (dtype != SSD_DTYPE_F32 && dtype != SSD_DTYPE_BF16) return SSD_ERR_INVALID_ARG;
  const int elt = dtype == SSD_DTYPE_BF16 ? 2 : 4;
  if (rows < 1 || cols < 1 || M < 1 || ((size_t)cols * elt) % 16) return SSD_ERR_INVALID_ARG;
  if (M > kMaxM || (rows + kRT - 1) / kRT > kNoAllocTiles) return SSD_ERR_CAPACITY;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SSD_ERR_CUDA;
  NoAllocDevice nd;
  {
    // once per device, with that device current: the array's device address
    // (the symbol's host-side name is not one), kernel attributes, SM count
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    NoAllocDevice& d = g_noalloc_dev[dev];
    if (!d.ready) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) return SSD_ERR_CUDA;
      if (prepare_gemv_kernels() != cudaSuccess) return SSD_ERR_CUDA;
      int sms = 0;
      if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return SSD_ERR_CUDA;
      d.scratch = static_cast<unsigned char*>(p);
      d.sms = sms < kNoAllocBlocks ? sms : kNoAllocBlocks;
      d.ready = true;
    }
    nd = d;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  Bufs B{};
  B.gpart = reinterpret_cast<float*>(nd.scratch);
  B.tile_counter = reinterpret_cast<uint32_t*>(nd.scratch + kNoAllocPart);
  B.ctl = reinterpret_cast<Ctl*>(nd.scratch + kNoAllocPart + kNoAllocCount);
  Dims D{};
  D.num_sms = nd.sms;
  // tickets and the error word start at zero on every call
  if (cudaMemsetAsync(B.tile_counter, 0, kNoAllocCount + kNoAllocCtl, st) != cudaSuccess)
    return SSD_ERR_CUDA;
  if (launch_gemv_plain(D, B, dtype, W, rows, cols, x_dev, M, y_dev, st) != cudaSuccess)
    return SSD_ERR_CUDA;
  // the error word a bounded wait sets when it gives up, for the caller to read
  if (err_dev && cudaMemcpyAsync(err_dev, &B.ctl->err, sizeof(int32_t), cudaMemcpyDeviceToDevice,
                                 st) != cudaSuccess)
    return SSD_ERR_CUDA;
  return SSD_OK;
}

namespace ssd {
// ----------------------------------------------------------------- probe
__global__ void k_read_probe(const uint4* __restrict__ src, uint64_t n16, uint32_t* sink) {
  uint32_t acc = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + 3 * stride < n16; i += 4 * stride) {
    const uint4 a = ld_stream16(src + i), b = ld_stream16(src + i + stride);
    const uint4 c = ld_stream16(src + i + 2 * stride), d = ld_stream16(src + i + 3 * stride);
    acc ^= a.x ^ a.y ^ a.z ^ a.w ^ b.x ^ b.y ^ b.z ^ b.w ^ c.x ^ c.y ^ c.z ^ c.w ^ d.x ^ d.y ^ d.z ^ d.w;
  }
  for (; i < n16; i += stride) {
    const uint4 a = ld_stream16(src + i);
    acc ^= a.x ^ a.y ^ a.z ^ a.w;
  }
  if (acc == 0x9E3779B9u) atomicXor(sink, acc);  // keeps the loads live
}

cudaError_t launch_read_probe(const void* src, uint64_t bytes, uint32_t* sink, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  k_read_probe<<<sms * 4, 512, 0, st>>>(static_cast<const uint4*>(src), bytes / 16, sink);
  return cudaGetLastError();
}

}  // namespace ssd
