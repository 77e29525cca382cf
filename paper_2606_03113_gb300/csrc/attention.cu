// attention.cu -- split-K decode attention over the contiguous KV cache for
// 1 (drafting, autoregressive) or k + 1 (verification) query rows, with GQA:
// k_attn (fp32 models, CUDA cores, one kernel) and k_attn_rows with
// k_attn_merge (bf16 models, tensor cores; below).
//
// k_attn: grid = (key splits of kAttnKeys, KV heads).  A block stages its keys and
// values once (fp32 in shared memory) and serves every query head of the KV
// group and every query row with them, so a GQA group of G heads and M rows
// share one KV read.  Row m sits at position pos0 + m and attends causally to
// keys [0, pos0 + m] (the new rows' own keys were appended by the QKV kernel).
//
// Keys before pos0 were written by earlier passes, so a block loads them
// before waiting for the QKV kernel that precedes it (programmatic dependent
// launch) and loads only the M new keys after the wait.  The row window
// (pos0, M) is read before the wait too: every writer of the control block
// runs at least one full dependency before this kernel is launched; it is
// read again after the wait and a mismatch is flagged and handled by
// reloading every key.
//
// Each (row, head, split) writes an unnormalised partial (max, sum, output);
// the last split block to finish a (KV head, row) pair -- a ticket per pair --
// merges its G heads' partials in split order with the log-sum-exp rule, so
// the result does not depend on which block finishes last.  A block that
// finishes several rows merges them all at once (verification passes).
#include <math.h>

#include "kernels.h"
#include "mma.cuh"
#include "pipe.cuh"

namespace ssd {

namespace {

constexpr int kAK = kAttnKeys;   // keys per split (two per lane)
constexpr int kAThreads = 256;
constexpr int kMergeBatch = 40;  // split partials loaded per round of the merge
constexpr int kMergeBatch4 = 8;  // ... four dimensions each, when merging many rows
constexpr int kAWarps = kAThreads / 32;

// Stages keys [k0, k1) of the split (relative to s0) into shared memory: the
// loads of a thread's kUnroll chunks are issued before any is stored.
__device__ __forceinline__ void stage_keys(const float* kb, const float* vb, int hd, int k0, int k1,
                                           float* Ks, float* Vs) {
  const int cpr = hd / 4;  // 16-byte chunks per key row
  const int n = (k1 - k0) * cpr;
  constexpr int kUnroll = 4;
  for (int c0 = threadIdx.x; c0 < n; c0 += kAThreads * kUnroll) {
    float4 ku[kUnroll], vu[kUnroll];
#pragma unroll
    for (int j = 0; j < kUnroll; ++j) {
      const int c = c0 + j * kAThreads;
      if (c < n) {
        const int key = k0 + c / cpr, off = (c % cpr) * 4;
        ku[j] = __ldg(reinterpret_cast<const float4*>(kb + (size_t)key * hd + off));
        vu[j] = __ldg(reinterpret_cast<const float4*>(vb + (size_t)key * hd + off));
      }
    }
#pragma unroll
    for (int j = 0; j < kUnroll; ++j) {
      const int c = c0 + j * kAThreads;
      if (c < n) {
        const int key = k0 + c / cpr, off = (c % cpr) * 4;
        float* kr = Ks + key * (hd + 1) + off;
        kr[0] = ku[j].x;
        kr[1] = ku[j].y;
        kr[2] = ku[j].z;
        kr[3] = ku[j].w;
        float* vr = Vs + key * hd + off;
        vr[0] = vu[j].x;
        vr[1] = vu[j].y;
        vr[2] = vu[j].z;
        vr[3] = vu[j].w;
      }
    }
  }
}

}  // namespace

// Three blocks per SM (the shared memory of a split allows three).
__global__ void __launch_bounds__(kAThreads, 3) k_attn(Dims D, Bufs B, int layer, RowSel sel) {
  extern __shared__ float sm[];
  const int split = blockIdx.x, g = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int hd = D.hd;
  const int G = D.Hq / D.Hkv;
  float* Ks = sm;                           // [kAK][hd + 1] (padded: lane-per-key reads)
  float* Vs = Ks + kAK * (hd + 1);          // [kAK][hd]
  float* Ps = Vs + kAK * hd;                // [warps][kAK] probabilities
  int* last_rows = reinterpret_cast<int*>(Ps + kAWarps * kAK);  // [kMaxM] rows this block merges
  __shared__ int s_nlast;

  const float* kv = static_cast<const float*>(B.kv) + (size_t)layer * 2 * D.Hkv * D.max_seq * hd;
  const int s0 = split * kAK;
  const float* kb = kv + ((size_t)g * D.max_seq + s0) * hd;
  const float* vb = kv + ((size_t)(D.Hkv + g) * D.max_seq + s0) * hd;

  // keys written by earlier passes: loaded before the wait
  int pos0, M;
  resolve_rows(B.ctl, sel, pos0, M);
  int nold = min(max(min(pos0, D.max_seq) - s0, 0), kAK);  // clamped: never past the cache
  if (pos0 + M > s0 && nold > 0) stage_keys(kb, vb, hd, 0, nold, Ks, Vs);
  pdl_wait();
  pdl_launch_dependents();
  {
    int p2, m2;
    resolve_rows(B.ctl, sel, p2, m2);
    if (p2 != pos0 || m2 != M) {  // the window moved: reload every key
      if (threadIdx.x == 0) atomicOr(&B.ctl->err, (int)kErrControl);
      pos0 = p2;
      M = m2;
      nold = 0;
    }
  }
  if (s0 > pos0 + M - 1) return;  // beyond every row's causal window
  const int nkeys = min(kAK, pos0 + M - s0);
  if (nkeys > nold) stage_keys(kb, vb, hd, nold, nkeys, Ks, Vs);
  __syncthreads();

  // partial attention of every (row, head) pair of the group over this split
  const float scale = 1.0f / sqrtf((float)hd);
  float* pw = Ps + warp * kAK;
  const int m_first = max(0, s0 - pos0);  // rows that see at least one key here
  const int npairs = G * (M - m_first);
  for (int pi = warp; pi < npairs; pi += kAWarps) {
    const int m = m_first + pi / G, qh = g * G + pi % G;
    const int pos = pos0 + m;
    const float* q = B.xq + (size_t)m * D.qd + (size_t)qh * hd;
    const int ka = lane, kb2 = lane + 32;
    const bool va = s0 + ka <= pos && ka < nkeys, vb2 = s0 + kb2 <= pos && kb2 < nkeys;
    float da = 0.f, db = 0.f;
    const float* kra = Ks + ka * (hd + 1);
    const float* krb = Ks + kb2 * (hd + 1);
    for (int i = 0; i < hd; i += 4) {
      const float4 qv = __ldg(reinterpret_cast<const float4*>(q + i));
      da = fmaf(qv.x, kra[i], da);
      da = fmaf(qv.y, kra[i + 1], da);
      da = fmaf(qv.z, kra[i + 2], da);
      da = fmaf(qv.w, kra[i + 3], da);
      db = fmaf(qv.x, krb[i], db);
      db = fmaf(qv.y, krb[i + 1], db);
      db = fmaf(qv.z, krb[i + 2], db);
      db = fmaf(qv.w, krb[i + 3], db);
    }
    const float sa = va ? da * scale : -INFINITY, sb = vb2 ? db * scale : -INFINITY;
    const float mx = warp_max(fmaxf(sa, sb));
    const float pa = va ? expf(sa - mx) : 0.f, pb = vb2 ? expf(sb - mx) : 0.f;
    const float l = warp_sum(pa + pb);
    pw[ka] = pa;
    pw[kb2] = pb;
    __syncwarp();
    // a row whose keys all lie in this split is finished here (its merge would
    // be one partial with weight 1)
    const bool whole = pos < kAK;
    const size_t pidx = ((size_t)m * D.Hq + qh) * D.nsplit + split;
    float* part = whole ? B.attn_out + (size_t)m * D.qd + (size_t)qh * hd : B.attn_part + pidx * hd;
    for (int dd = lane; dd < hd; dd += 32) {
      float o = 0.f;
#pragma unroll 8
      for (int s = 0; s < nkeys; ++s) o = fmaf(pw[s], Vs[s * hd + dd], o);
      part[dd] = whole ? o / l : o;
    }
    if (lane == 0 && !whole) {
      B.attn_ml[2 * pidx] = mx;
      B.attn_ml[2 * pidx + 1] = l;
    }
    __syncwarp();
  }

  // tickets: the last split of (g, m) merges the group's heads for row m.
  // One thread per row takes the ticket with an acquire-release add after
  // the block barrier, which publishes the block's partials and, for the
  // last split, makes every other split's visible to the whole block.
  if (pos0 + M - 1 < kAK) return;  // every row is finished
  if (threadIdx.x == 0) s_nlast = 0;
  __syncthreads();
  if (threadIdx.x < M && threadIdx.x >= m_first && pos0 + (int)threadIdx.x >= kAK) {
    const int m = threadIdx.x;
    const int nsp = (pos0 + m) / kAK + 1;
    uint32_t* cnt = B.attn_counter + (size_t)g * kMaxM + m;
    if (atom_add_acq_rel_gpu(cnt, 1u) == (uint32_t)(nsp - 1)) {
      *cnt = 0u;
      last_rows[atomicAdd(&s_nlast, 1)] = m;
    }
  }
  __syncthreads();
  const int nlast = s_nlast;
  if (nlast == 0) return;
  // merge of every row this block finishes, all rows at once (the key and
  // value buffers are free now): (max, sum) of every (row, head, split) in
  // one round of loads, then the weights e^{m_s - max} and denominators (a
  // warp per (row, head), fixed lane order), then the outputs, each the
  // splits' partials added in split order)
  const int NS = D.nsplit;
  float* Cm = Ks;                                  // [nlast][G][NS] maxima
  float* Cw = Cm + (size_t)nlast * G * NS;         // [nlast][G][NS] sums, then weights
  float* CL = Cw + (size_t)nlast * G * NS;         // [nlast][G] denominators
  const int npr = nlast * G;
  for (int i = threadIdx.x; i < npr * NS; i += kAThreads) {
    const int pr = i / NS, sp = i - pr * NS;
    const int m = last_rows[pr / G], h = pr - (pr / G) * G;
    if (sp > (pos0 + m) / kAK) continue;
    const size_t pidx = ((size_t)m * D.Hq + (size_t)g * G + h) * NS + sp;
    Cm[i] = __ldcg(&B.attn_ml[2 * pidx]);
    Cw[i] = __ldcg(&B.attn_ml[2 * pidx + 1]);
  }
  __syncthreads();
  for (int pr = warp; pr < npr; pr += kAWarps) {
    const int m = last_rows[pr / G];
    const int nsp = (pos0 + m) / kAK + 1;
    const float* cm = Cm + (size_t)pr * NS;
    float* cw = Cw + (size_t)pr * NS;
    float gmax = -INFINITY;
    for (int sp = lane; sp < nsp; sp += 32) gmax = fmaxf(gmax, cm[sp]);
    gmax = warp_max(gmax);
    float L = 0.f;
    for (int sp = lane; sp < nsp; sp += 32) {
      const float l = cw[sp];
      const float w = l > 0.f ? expf(cm[sp] - gmax) : 0.f;
      cw[sp] = w;
      L = fmaf(w, l, L);
    }
    L = warp_sum(L);
    if (lane == 0) CL[pr] = L;
  }
  __syncthreads();
  if (npr * hd <= kAThreads) {
    // few rows: a thread per output, all splits in one round
    for (int o = threadIdx.x; o < npr * hd; o += kAThreads) {
      const int pr = o / hd, dd = o - pr * hd;
      const int m = last_rows[pr / G], h = pr - (pr / G) * G;
      const int nsp = (pos0 + m) / kAK + 1;
      const float* w = Cw + (size_t)pr * NS;
      const float* part = B.attn_part + (((size_t)m * D.Hq + (size_t)g * G + h) * NS) * hd + dd;
      float O = 0.f;
      for (int sc = 0; sc < nsp; sc += kMergeBatch) {
        float pv[kMergeBatch];
#pragma unroll
        for (int j = 0; j < kMergeBatch; ++j)
          pv[j] = sc + j < nsp ? __ldcg(part + (size_t)(sc + j) * hd) : 0.f;
#pragma unroll
        for (int j = 0; j < kMergeBatch; ++j)
          if (sc + j < nsp) O = fmaf(w[sc + j], pv[j], O);
      }
      B.attn_out[(size_t)m * D.qd + (size_t)(g * G + h) * hd + dd] = O / CL[pr];
    }
  } else {
    // many rows (verification): a warp per (row, head), four dimensions per
    // lane; the same sum per output, fewer rounds of loads
    for (int pr = warp; pr < npr; pr += kAWarps) {
      const int m = last_rows[pr / G], h = pr - (pr / G) * G;
      const int nsp = (pos0 + m) / kAK + 1;
      const float* w = Cw + (size_t)pr * NS;
      const float* part = B.attn_part + (((size_t)m * D.Hq + (size_t)g * G + h) * NS) * hd;
      float* out = B.attn_out + (size_t)m * D.qd + (size_t)(g * G + h) * hd;
      for (int d0 = 4 * lane; d0 < hd; d0 += 128) {
        float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int sc = 0; sc < nsp; sc += kMergeBatch4) {
          float4 pv[kMergeBatch4];
#pragma unroll
          for (int j = 0; j < kMergeBatch4; ++j)
            pv[j] = sc + j < nsp
                        ? __ldcg(reinterpret_cast<const float4*>(part + (size_t)(sc + j) * hd + d0))
                        : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int j = 0; j < kMergeBatch4; ++j)
            if (sc + j < nsp) {
              const float wj = w[sc + j];
              O.x = fmaf(wj, pv[j].x, O.x);
              O.y = fmaf(wj, pv[j].y, O.y);
              O.z = fmaf(wj, pv[j].z, O.z);
              O.w = fmaf(wj, pv[j].w, O.w);
            }
        }
        const float L = CL[pr];
        *reinterpret_cast<float4*>(out + d0) = make_float4(O.x / L, O.y / L, O.z / L, O.w / L);
      }
    }
  }
}

size_t attn_smem(const Dims& D) {
  // keys and values of one split (reused by the merge: maxima, weights and
  // denominators of up to kMaxM rows x G heads x nsplit splits), the warps'
  // probabilities, the rows this block merges
  const int G = D.Hq / D.Hkv;
  const size_t kv = (size_t)kAK * (D.hd + 1) + (size_t)kAK * D.hd;
  const size_t merge = (2 * (size_t)D.nsplit + 1) * kMaxM * G;
  return sizeof(float) * ((kv > merge ? kv : merge) + (size_t)kAWarps * kAK) + sizeof(int) * kMaxM;
}

// ------------------------------------------------------------ bf16 models
//
// k_attn_rows: block = (split of D.attn_keys keys, KV head); its keys and
// values are staged once as bf16 and serve the group's G x M query rows, 16
// rows at a time per group of four warps.  Scores and outputs run on
// mma.sync; the fp32 operand (queries, probabilities) enters in three bf16
// parts, 24 bits, so nothing is rounded below fp32.  Of a 64-key step a warp
// scores 16 keys; the four warps then share the row maxima and the
// probabilities through shared memory and each multiplies all 64 keys with
// its 32 of the 128 output columns.  A row's sums depend on its position
// alone, not on the number of rows or on the other rows of its tile.
// k_attn_merge: a warp per (row, head) adds the splits' partials in split
// order.  A launch of its own: the last block of a KV head used to merge
// alone, 136 rows x 17 splits in the widest verification.
//
// Bound by the chain of load, score, exchange, multiply within a block (the
// KV rows are 1 to 45 MB).  us a call against the earlier kernel on CUDA
// cores (one warp per (row, head) pair and 64 keys, merge by the last block):
// 13 rows of the 8B widths after 1100 tokens, 4 layers, 1276 to 974; 17 rows
// (70B, 1024 tokens, 2 layers) 1336 to 937; 2 rows (13B, 2176 tokens, 4
// layers) 886 to 800; one row (7B, 640 tokens, 4 layers) 603 to 572.

namespace {

constexpr int kRHd = 128;
constexpr int kRStep = kAttnKeys;                    // keys per step
constexpr int kRGThreads = 128;                      // a row group: four warps
constexpr int kRMaxGroups = 4;
constexpr size_t kRKeyBytes = (size_t)kRStep * kRHd * 2;      // keys (or values) of a step
constexpr size_t kRQBytes = (size_t)3 * 16 * kRHd * 2;        // 16 query rows, three parts
constexpr size_t kRPBytes = (size_t)3 * 16 * kRStep * 2;      // their probabilities
constexpr size_t kRGroupBytes = kRQBytes + kRPBytes + 2 * 4 * 16 * sizeof(float);

}  // namespace

__global__ void __launch_bounds__(kRGThreads * kRMaxGroups)
    k_attn_rows(const Dims D, const Bufs B, int layer, RowSel sel) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int split = blockIdx.x, g = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31;
  const int rg = tid / kRGThreads, ngrp = (int)blockDim.x / kRGThreads;
  const int w = (tid >> 5) & 3;
  const int G = D.Hq / D.Hkv;
  const int len = D.attn_keys, s0 = split * len;
  const __nv_bfloat16* kv =
      static_cast<const __nv_bfloat16*>(B.kv) + (size_t)layer * 2 * D.Hkv * D.max_seq * kRHd;
  const __nv_bfloat16* kb = kv + ((size_t)g * D.max_seq + s0) * kRHd;
  const __nv_bfloat16* vb = kv + ((size_t)(D.Hkv + g) * D.max_seq + s0) * kRHd;
  const uint32_t sbase = smem_u32(smem);

  // keys [k0, k1) of the split; those from kend on are filled with zeros
  auto stage = [&](int k0, int k1, int kend) {
    for (int c = tid; c < (k1 - k0) * 16; c += (int)blockDim.x) {
      const int key = k0 + (c >> 4), ch = c & 15;
      const bool in = key < kend;
      const size_t off = (size_t)(in ? key : 0) * kRHd + ch * 8;
      const uint32_t dst = sbase + (uint32_t)(key / kRStep) * (uint32_t)(2 * kRKeyBytes) +
                           sw256(key % kRStep, ch);
      cp_async16(dst, kb + off, in);
      cp_async16(dst + (uint32_t)kRKeyBytes, vb + off, in);
    }
  };

  // keys written by earlier passes: loaded before the wait
  int pos0, M;
  resolve_rows(B.ctl, sel, pos0, M);
  int nold = min(max(min(pos0, D.max_seq) - s0, 0), len);  // clamped: never past the cache
  if (pos0 + M <= s0) nold = 0;
  stage(0, nold, nold);
  pdl_wait();
  pdl_launch_dependents();
  {
    int p2, m2;
    resolve_rows(B.ctl, sel, p2, m2);
    if (p2 != pos0 || m2 != M) {  // the window moved: reload every key
      if (tid == 0) atomicOr(&B.ctl->err, (int)kErrControl);
      cp_async_wait_all();
      __syncthreads();
      pos0 = p2;
      M = m2;
      nold = 0;
    }
  }
  if (s0 > pos0 + M - 1) {  // beyond every row's causal window
    cp_async_wait_all();
    return;
  }
  const int nkeys = min(len, pos0 + M - s0);
  const int nsteps = (nkeys + kRStep - 1) / kRStep;
  stage(nold, nsteps * kRStep, nkeys);

  unsigned char* grp = smem + (size_t)(len / kRStep) * 2 * kRKeyBytes + (size_t)rg * kRGroupBytes;
  const uint32_t qs = smem_u32(grp), ps = qs + (uint32_t)kRQBytes;
  float* smx = reinterpret_cast<float*>(grp + kRQBytes + kRPBytes);  // [warp][row] maxima
  float* sls = smx + 4 * 16;                                         // [warp][row] sums
  const int gt = tid % kRGThreads;
  const float scale = 1.0f / sqrtf((float)kRHd);
  const int row_lo = max(0, s0 - pos0) * G, nrows = G * M;  // rows that see a key here
  const int rr = lane >> 2;  // the thread's rows of a tile: rr and rr + 8
  bool staged = false;

  for (int r0 = row_lo + 16 * rg; r0 < nrows; r0 += 16 * ngrp) {
    // queries of the tile: three bf16 parts (rows past the last are zero)
    for (int c = gt; c < 16 * 16; c += kRGThreads) {
      const int row = c >> 4, ch = c & 15, r = r0 + row;
      float4 x0 = make_float4(0.f, 0.f, 0.f, 0.f), x1 = x0;
      if (r < nrows) {
        const int m = r / G, h = g * G + r - m * G;
        const float4* p =
            reinterpret_cast<const float4*>(B.xq + (size_t)m * D.qd + (size_t)h * kRHd + ch * 8);
        x0 = p[0];
        x1 = p[1];
      }
      uint4 q3[3];
      split3(x0.x, x0.y, q3[0].x, q3[1].x, q3[2].x);
      split3(x0.z, x0.w, q3[0].y, q3[1].y, q3[2].y);
      split3(x1.x, x1.y, q3[0].z, q3[1].z, q3[2].z);
      split3(x1.z, x1.w, q3[0].w, q3[1].w, q3[2].w);
#pragma unroll
      for (int s = 0; s < 3; ++s)
        *reinterpret_cast<uint4*>(grp + (size_t)s * 16 * 256 + sw256(row, ch)) = q3[s];
    }
    if (!staged) {
      cp_async_wait_all();
      __syncthreads();
      staged = true;
    } else {
      named_sync(1 + rg, kRGThreads);
    }
    int pos[2];
    float mx[2], ls[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int r = r0 + rr + 8 * e;
      pos[e] = r < nrows ? pos0 + r / G : s0;  // an unused row sees the split's first key
      mx[e] = -INFINITY;
      ls[e] = 0.f;
    }
    float o[4][4];
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[n][e] = 0.f;

    for (int st = 0; st < nsteps; ++st) {
      const uint32_t kd = sbase + (uint32_t)st * (uint32_t)(2 * kRKeyBytes);
      const uint32_t vd = kd + (uint32_t)kRKeyBytes;
      // scores of the warp's 16 keys: two n-tiles, even and odd 16-column
      // steps summed apart; the lower parts first, since the running sum is
      // cut at its own last place
      float s[2][2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
          for (int e = 0; e < 4; ++e) s[i][n][e] = 0.f;
#pragma unroll
      for (int pass = 0; pass < 2; ++pass)
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          uint32_t kf[4];
          ldsm4(kd + sw256(16 * w + (lane & 7) + ((lane >> 4) << 3), 2 * kk + ((lane >> 3) & 1)), kf);
#pragma unroll
          for (int p = pass ? 0 : 2; p >= (pass ? 0 : 1); --p) {
            uint32_t qa[4];
            ldsm4(qs + (uint32_t)(p * 16 * 256) + sw256(lane & 15, 2 * kk + (lane >> 4)), qa);
            mma16816(s[kk & 1][0], qa, kf[0], kf[1]);
            mma16816(s[kk & 1][1], qa, kf[2], kf[3]);
          }
        }
      const int kbase = s0 + st * kRStep + 16 * w + 2 * (lane & 3);
      float z[2][4], nm[2] = {-INFINITY, -INFINITY};
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int key = kbase + 8 * n + (e & 1);
          z[n][e] = key <= pos[e >> 1] ? (s[0][n][e] + s[1][n][e]) * scale : -INFINITY;
          nm[e >> 1] = fmaxf(nm[e >> 1], z[n][e]);
        }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        nm[e] = fmaxf(nm[e], __shfl_xor_sync(0xffffffffu, nm[e], 1));
        nm[e] = fmaxf(nm[e], __shfl_xor_sync(0xffffffffu, nm[e], 2));
        if ((lane & 3) == 0) smx[w * 16 + rr + 8 * e] = nm[e];
      }
      named_sync(1 + rg, kRGThreads);
      float f[2], rs[2] = {0.f, 0.f};
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float m = mx[e];
#pragma unroll
        for (int i = 0; i < 4; ++i) m = fmaxf(m, smx[i * 16 + rr + 8 * e]);
        // every row sees the split's first key: finite from the first step on
        f[e] = expf(mx[e] - m);
        mx[e] = m;
      }
#pragma unroll
      for (int n = 0; n < 2; ++n) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          z[n][e] = expf(z[n][e] - mx[e >> 1]);
          rs[e >> 1] += z[n][e];
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          uint32_t q[3];
          split3(z[n][2 * e], z[n][2 * e + 1], q[0], q[1], q[2]);
#pragma unroll
          for (int p = 0; p < 3; ++p)
            *reinterpret_cast<uint32_t*>(grp + kRQBytes + (size_t)p * 16 * 128 +
                                         sw128(rr + 8 * e, 2 * w + n) + 4 * (lane & 3)) = q[p];
        }
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        rs[e] += __shfl_xor_sync(0xffffffffu, rs[e], 1);
        rs[e] += __shfl_xor_sync(0xffffffffu, rs[e], 2);
        if ((lane & 3) == 0) sls[w * 16 + rr + 8 * e] = rs[e];
      }
      named_sync(1 + rg, kRGThreads);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float* l = sls + rr + 8 * e;
        ls[e] = fmaf(ls[e], f[e], (l[0] + l[16]) + (l[32] + l[48]));
      }
      // outputs: columns 32 w .. 32 w + 31, this step's share in sums of its
      // own, then one rounded multiply-add into the running output
      float t[4][4];
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) t[n][e] = 0.f;
#pragma unroll
      for (int p = 2; p >= 0; --p)
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          uint32_t pa[4];
          ldsm4(ps + (uint32_t)(p * 16 * 128) + sw128(lane & 15, 2 * ks + (lane >> 4)), pa);
#pragma unroll
          for (int n2 = 0; n2 < 2; ++n2) {
            uint32_t vf[4];
            ldsm4t(vd + sw256(16 * ks + (lane & 15), 4 * w + 2 * n2 + (lane >> 4)), vf);
            mma16816(t[2 * n2], pa, vf[0], vf[1]);
            mma16816(t[2 * n2 + 1], pa, vf[2], vf[3]);
          }
        }
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[n][e] = fmaf(o[n][e], f[e >> 1], t[n][e]);
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int r = r0 + rr + 8 * e;
      if (r >= nrows) continue;
      const int m = r / G, h = g * G + r - m * G;
      const size_t pidx = ((size_t)m * D.Hq + h) * D.nsplit + split;
      float* part = B.attn_part + pidx * kRHd + 32 * w + 2 * (lane & 3);
#pragma unroll
      for (int n = 0; n < 4; ++n)
        *reinterpret_cast<float2*>(part + 8 * n) = make_float2(o[n][2 * e], o[n][2 * e + 1]);
      if (w == 0 && (lane & 3) == 0)
        *reinterpret_cast<float2*>(B.attn_ml + 2 * pidx) = make_float2(mx[e], ls[e]);
    }
  }
  if (!staged) {  // a group without rows: the others' barrier
    cp_async_wait_all();
    __syncthreads();
  }
}

// Merge of the splits: a warp per (row, head), four columns per lane.
__global__ void __launch_bounds__(256) k_attn_merge(const Dims D, const Bufs B, RowSel sel) {
  pdl_wait();
  pdl_launch_dependents();
  int pos0, M;
  resolve_rows(B.ctl, sel, pos0, M);
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int m = i / D.Hq;
  if (m >= M) return;
  const int nsp = (pos0 + m) / D.attn_keys + 1;
  const float2* ml = reinterpret_cast<const float2*>(B.attn_ml) + (size_t)i * D.nsplit;
  const float4* part =
      reinterpret_cast<const float4*>(B.attn_part + (size_t)i * D.nsplit * kRHd) + lane;
  constexpr int kBatch = 8;
  float gmax = -INFINITY;
  for (int s = lane; s < nsp; s += 32) gmax = fmaxf(gmax, __ldcg(&ml[s]).x);
  gmax = warp_max(gmax);
  float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
  float L = 0.f;
  for (int s0 = 0; s0 < nsp; s0 += kBatch) {
    float4 p[kBatch];
    float2 a[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const int s = s0 + j < nsp ? s0 + j : s0;
      p[j] = __ldcg(part + (size_t)s * (kRHd / 4));
      a[j] = __ldcg(&ml[s]);
    }
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const float wj = s0 + j < nsp ? expf(a[j].x - gmax) : 0.f;
      L = fmaf(wj, a[j].y, L);
      O.x = fmaf(wj, p[j].x, O.x);
      O.y = fmaf(wj, p[j].y, O.y);
      O.z = fmaf(wj, p[j].z, O.z);
      O.w = fmaf(wj, p[j].w, O.w);
    }
  }
  // as the O projection reads it
  uint2 hi, lo;
  split2(O.x / L, O.y / L, hi.x, lo.x);
  split2(O.z / L, O.w / L, hi.y, lo.y);
  __nv_bfloat16* xo = B.xs_o + (size_t)i * kRHd + 4 * lane;
  *reinterpret_cast<uint2*>(xo) = hi;
  *reinterpret_cast<uint2*>(xo + (size_t)kMaxM * D.qd) = lo;
}

// Keys per split of the bf16 kernel: 64, or 128 where 64 would make more blocks
// than three per SM with a full cache: fewer partials to store and merge, for
// two key steps in a row.  One value for a model's whole cache, since a row's
// sums have to be the same in drafting and in verification.  Live with the merge,
// a cache of 2304 positions, us a layer for 1 / 17 rows with 128 and 64 keys:
//   context             100                     1000                    2176
//   32 KV heads   7.5/10.3, 7.0/9.4       9.2/13.1, 10.6/16.2    17.1/23.1, 18.2/27.9
//   40 KV heads   7.8/10.9, 7.2/10.1     11.3/16.4, 12.0/18.9    21.2/28.5, 20.3/32.8
//    8 (of 64)    6.2/20.5, 6.0/15.4      6.4/21.3,  7.3/18.7     8.8/24.5, 10.7/33.3
// So 128 loses 5 to 10 % at the beginning of a long cache and 4 % for one row
// of 40 heads behind 2048 positions, and wins up to 20 % elsewhere.  With few
// KV heads (the last line, which the rule gives 64) a wide verification is a
// third faster with 64 up to some 640 positions and as much slower from 1500
// on; there the rule keeps the shorter contexts' choice.
int attn_split_keys(int n_kv_heads, int max_seq, int sms) {
  const int n = (max_seq + kRStep - 1) / kRStep;
  return n_kv_heads * n > 3 * sms ? 2 * kRStep : kRStep;
}

static size_t rows_smem(int keys, int groups) {
  return (size_t)(keys / kRStep) * 2 * kRKeyBytes + groups * kRGroupBytes;
}

// The limits of dynamic shared memory, once and the same for every context: a
// function's attributes are shared by all threads, and a launch's own size
// depends on the model and on the number of rows.
cudaError_t prepare_attention_kernels(int dtype) {
  if (dtype == SSD_DTYPE_BF16)
    return cudaFuncSetAttribute(k_attn_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)rows_smem(2 * kRStep, kRMaxGroups));
  // what the device has: the merge of a long cache takes more than a split's keys
  int dev = 0, most = 0;
  cudaFuncAttributes fa;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_attn);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_attn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              most - (int)fa.sharedSizeBytes);
}

static cudaError_t attn_bf16(const Dims& D, const Bufs& B, int layer, RowSel sel, int mrows,
                             cudaStream_t st) {
  const int rows = mrows * (D.Hq / D.Hkv);
  const int groups = rows <= 16 ? 1 : (rows <= 32 ? 2 : kRMaxGroups);
  const size_t smem = rows_smem(D.attn_keys, groups);
  const dim3 grid((D.max_seq + D.attn_keys - 1) / D.attn_keys, D.Hkv);
  cudaError_t e = launch_ex(k_attn_rows, grid, dim3(groups * kRGThreads), smem, st, D, B, layer, sel);
  if (e != cudaSuccess) return e;
  return launch_ex(k_attn_merge, dim3((mrows * D.Hq + 7) / 8), dim3(256), 0, st, D, B, sel);
}

static cudaError_t attn_f32(const Dims& D, const Bufs& B, int layer, RowSel sel, cudaStream_t st) {
  dim3 grid(D.nsplit, D.Hkv);
  return launch_ex(k_attn, grid, dim3(kAThreads), attn_smem(D), st, D, B, layer, sel);
}

cudaError_t launch_attention(const Dims& D, const Bufs& B, int dtype, int layer, RowSel sel,
                             int mrows, cudaStream_t st) {
  if (dtype == SSD_DTYPE_BF16) return attn_bf16(D, B, layer, sel, mrows, st);
  return attn_f32(D, B, layer, sel, st);
}

}  // namespace ssd
