// Prompt-wide base scores on the tensor cores (bf16): the Mean Attention and
// full-attention ("snapshot") bases of the base-scoring ablation (appendix
// "Sensitivity to the Base Attention Scoring Function").  The last nq cached
// positions are query rows; row (position p, query head g) attends causally
// to keys j <= p.  For KV head h:
//   C[j] = (1/G) sum_{g in group h} sum_{p >= j} softmax_{j' <= p}(q_{p,g} . k_{j',h} / sqrt(d))_j
// full base A = C; Mean Attention A = C / #{prompt rows that attend to j}.
//
//   k_prompt_rowstats  pass 1: persistent CTAs over the 128-row m-tiles of
//                      query rows (P1 = floor(128 / G) whole positions, G rows
//                      each), longest first; per m-tile key tiles of 256
//                      stream up to its last position; per row the running
//                      max and sum of exponentials under the causal mask,
//                      merged over four epilogue groups into bias_r = -m_r -
//                      log2(G l_r).
//   k_prompt_colsum    pass 2: a cluster of CTAs per 128-key tile, the tile
//                      resident in shared memory as the A operand; chunks of
//                      P2 = floor(256 / G) positions (G P2 rows) stream as the
//                      B operand from the first chunk that can see the tile,
//                      the cluster's CTAs taking them in turn; each key sums
//                      2^(x c + bias_r) over the rows that attend to it, and
//                      the CTAs' sums are added in rank order: no atomics, no
//                      reduction pass.
//
// Query rows come straight from q [nq][Hq][128] through a 3-D TMA box (d,
// the group's G heads, positions): its lines land in shared memory in
// (position, head) order, which is the row order r = position * G + g.
// Same warp roles as the window-score passes: warp 0 TMA, warp 1 MMA, four
// groups of four epilogue warps; every mbarrier wait is bounded.
//
// Both passes are bound by their epilogues (0.9 and 1.1 us per 128 x 256 item,
// the MMA alone 0.66).  8,576 positions, 28 query heads (one layer), with one
// CTA per m-tile and per key tile, the biases in the query rows' stages and a
// kernel that filled the bias array first: 6 + 210 + 255 us; now 187 + 241.
#include <cooperative_groups.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>

#include "kernels.cuh"
#include "ptx.cuh"
#include "tile.cuh"

namespace cg = cooperative_groups;

namespace stl {

namespace {

constexpr int kPrGroups = 4;
constexpr int kPrThreads = (2 + 4 * kPrGroups) * 32;
constexpr int kPrMaxReg = 96;
constexpr float kPrLog2e = 1.4426950408889634f;

// pass 1: two Q m-tiles [2 halves][128 rows][128 B] (the next one loads
// while this one is worked on), two key stages of 256 keys
constexpr int kP1Q = 0;
constexpr int kP1K = 2 * 32768;
constexpr int kP1KStage = 65536;
constexpr int kP1Stages = 2;
constexpr int kP1Bar = kP1K + kP1Stages * kP1KStage;  // 13 mbarriers, slot, abort
constexpr int kP1Xch = kP1Bar + 128;                   // float2 [2][4 groups][128 rows]
constexpr int kP1Smem = kP1Xch + 2 * kPrGroups * 128 * 8 + 1024;

// pass 2: key tile [2 halves][128 keys][128 B], two Q stages of 256 rows,
// four stages of row biases, the groups' partial sums, the CTA's sums
constexpr int kP2K = 0;
constexpr int kP2Q = 32768;
constexpr int kP2QStage = 65536;
constexpr int kP2Stages = 2;
constexpr int kP2BStages = 4;
constexpr int kP2Bias = kP2Q + kP2Stages * kP2QStage;  // float [stages][256]
constexpr int kP2Bar = kP2Bias + kP2BStages * 1024;    // 18 mbarriers, slot, abort
constexpr int kP2Xch = kP2Bar + 256;                    // float [4 groups][128 keys]
constexpr int kP2Sum = kP2Xch + kPrGroups * 128 * 4;    // float2 [128 keys]
constexpr int kP2Smem = kP2Sum + 128 * 8 + 1024;
constexpr int kP2MaxSplit = 8;                          // CTAs per key tile (one cluster)

__device__ __forceinline__ uint8_t* pr_align1024(uint8_t* p) {
  uint32_t a = smem_u32(p);
  return p + ((1024u - (a & 1023u)) & 1023u);
}

// Contiguous global -> shared copy completing on `bar` (16-byte aligned
// addresses, size a multiple of 16).
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar)
               : "memory");
}

// Named barrier over the 16 epilogue warps (id 1).
__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 1, %0;" ::"n"(4 * kPrGroups * 32)); }

}  // namespace

struct PromptMaps {
  CUtensorMap q1;  // box 64 x G x P1
  CUtensorMap q2;  // box 64 x G x P2
  CUtensorMap k1;  // box 64 x 1 x 256
  CUtensorMap k2;  // box 64 x 1 x 128
};

struct PromptArgs {
  int n, nq, hq, hkv, G;
  int p1, p2;      // positions per pass-1 m-tile / pass-2 chunk
  int n_mt, n_ch;  // m-tiles and chunks per head
  int crp;         // bias floats per chunk (G P2 rounded up to 4)
  int mode;        // 0 full, 1 mean
};

// bias [Hkv][n_ch][crp]: entry of row (relative position pr, head g of the
// group) at chunk pr / P2, offset (pr % P2) G + g; every other entry -inf.
// Those others: the ends of the chunks' rows, and the last chunk's positions
// past the prompt (a few values per chunk, shared out over the grid).
__device__ __forceinline__ void prompt_bias_pad(const PromptArgs& a, float* bias) {
  for (int c = blockIdx.x; c < a.hkv * a.n_ch; c += gridDim.x) {
    const int real = a.G * min(a.p2, a.nq - c % a.n_ch * a.p2);
    for (int i = real + threadIdx.x; i < a.crp; i += blockDim.x) bias[(size_t)c * a.crp + i] = -CUDART_INF_F;
  }
}

__global__ void __maxnreg__(kPrMaxReg)
    k_prompt_rowstats(const __grid_constant__ PromptMaps maps, PromptArgs a, float* bias, uint32_t* err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = pr_align1024(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // work item i: KV head i % hkv, m-tile n_mt - 1 - i / hkv (longest rows
  // first).  The CTAs take a grid's worth of items per round, in turn from the
  // first to the last CTA and back: always in the same order, the first CTA
  // had 16 % more keys than the last (8,576 positions: 197 us, now 187).  An
  // item's rows are positions [pr0, pr0 + npos), its keys [0, p_first + pr0 +
  // npos).
  const int n_items = a.n_mt * a.hkv, p_first = a.n - a.nq;
  auto item = [&](int round) {
    return round * (int)gridDim.x + (int)(round & 1 ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
  };
  auto item_pr0 = [&](int i) { return (a.n_mt - 1 - i / a.hkv) * a.p1; };
  auto item_tiles = [&](int pr0) { return (p_first + pr0 + min(a.p1, a.nq - pr0) + 255) / 256; };
  const uint32_t sQ = smem_u32(sm + kP1Q), sK = smem_u32(sm + kP1K);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + kP1Bar);
  const uint32_t b_kfull = smem_u32(&bars[0]), b_kempty = smem_u32(&bars[kP1Stages]);
  const uint32_t b_accfull = smem_u32(&bars[2 * kP1Stages]), b_accempty = smem_u32(&bars[2 * kP1Stages + 2]);
  const uint32_t b_qfull = smem_u32(&bars[2 * kP1Stages + 4]), b_qempty = smem_u32(&bars[2 * kP1Stages + 6]);
  const uint32_t b_done = smem_u32(&bars[2 * kP1Stages + 8]);
  uint32_t* slot = reinterpret_cast<uint32_t*>(sm + kP1Bar + 8 * (2 * kP1Stages + 9));
  volatile uint32_t* abort_flag = slot + 1;
  float2* xch = reinterpret_cast<float2*>(sm + kP1Xch);
  const float c = kPrLog2e * rsqrtf((float)kD);

  if (threadIdx.x == 0) {
    for (int i = 0; i < kP1Stages; ++i) {
      mbar_init(b_kfull + 8 * i, 1);
      mbar_init(b_kempty + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(b_accfull + 8 * i, 1);
      mbar_init(b_accempty + 8 * i, 4 * kPrGroups);
      mbar_init(b_qfull + 8 * i, 1);
      mbar_init(b_qempty + 8 * i, 1);
    }
    mbar_init(b_done, 1);
    *abort_flag = 0u;
    fence_mbar_init();
    tma_prefetch_desc(&maps.q1);
    tma_prefetch_desc(&maps.k1);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(slot), 512);
    tmem_relinquish();
  }
  prompt_bias_pad(a, bias);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;

  if (warp == 0) {
    if (lane == 0) {
      // an item's rows: positions [pr0, pr0 + P1) of the group's G heads
      const uint32_t qbytes = 2u * 128u * (uint32_t)(a.G * a.p1);
      int issued[kP1Stages] = {0, 0}, q_issued[2] = {0, 0};
      int ks = 0, qi = 0;  // key stage; items so far
      uint32_t kp = 0u;
      bool ok = true;
      for (int i = item(0); ok && i < n_items; i = item(++qi)) {
        const int qs = qi & 1, h = i % a.hkv, pr0 = item_pr0(i), ntiles = item_tiles(pr0);
        if (!mbar_wait(b_qempty + 8 * qs, ((uint32_t)(qi >> 1) & 1u) ^ 1u, err, abort_flag)) break;
        mbar_arrive_expect_tx(b_qfull + 8 * qs, qbytes);
        tma_load_3d(sQ + qs * 32768, &maps.q1, b_qfull + 8 * qs, 0, h * a.G, pr0);
        tma_load_3d(sQ + qs * 32768 + 16384, &maps.q1, b_qfull + 8 * qs, 64, h * a.G, pr0);
        ++q_issued[qs];
        for (int it = 0; it < ntiles; ++it, ks = ks + 1 == kP1Stages ? 0 : ks + 1, kp += ks == 0 ? 1u : 0u) {
          if (!mbar_wait(b_kempty + 8 * ks, (kp & 1u) ^ 1u, err, abort_flag)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(b_kfull + 8 * ks, (uint32_t)kP1KStage);
          tma_load_3d(sK + ks * kP1KStage, &maps.k1, b_kfull + 8 * ks, 0, h, it * 256);
          tma_load_3d(sK + ks * kP1KStage + 32768, &maps.k1, b_kfull + 8 * ks, 64, h, it * 256);
          ++issued[ks];
        }
      }
      if (*abort_flag) {
        for (int s = 0; s < 2; ++s)
          if (q_issued[s]) mbar_wait_drain(b_qfull + 8 * s, (uint32_t)(q_issued[s] - 1) & 1u);
        for (int s = 0; s < kP1Stages; ++s)
          if (issued[s]) mbar_wait_drain(b_kfull + 8 * s, (uint32_t)(issued[s] - 1) & 1u);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16(128, 256);
      bool ok = true;
      int ks = 0, qi = 0, u = 0;  // key stage; items, key tiles so far
      uint32_t kp = 0u;
      for (int i = item(0); ok && i < n_items; i = item(++qi)) {
        const int qs = qi & 1, ntiles = item_tiles(item_pr0(i));
        if (!mbar_wait(b_qfull + 8 * qs, (uint32_t)(qi >> 1) & 1u, err, abort_flag)) break;
        for (int it = 0; it < ntiles;
             ++it, ++u, ks = ks + 1 == kP1Stages ? 0 : ks + 1, kp += ks == 0 ? 1u : 0u) {
          const int as = u & 1;
          if (!mbar_wait(b_kfull + 8 * ks, kp & 1u, err, abort_flag) ||
              !mbar_wait(b_accempty + 8 * as, ((uint32_t)(u >> 1) & 1u) ^ 1u, err, abort_flag)) {
            ok = false;
            break;
          }
          tc_fence_after();
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint32_t kb = k >> 2, koff = (k & 3) * 32;
            const uint64_t ad = desc_sw128(sQ + qs * 32768 + kb * 16384 + koff);
            const uint64_t bd = desc_sw128(sK + ks * kP1KStage + kb * 32768 + koff);
            umma_bf16(tmem + as * 256, ad, bd, idesc, k > 0 ? 1u : 0u);
          }
          umma_commit(b_accfull + 8 * as);
          umma_commit(b_kempty + 8 * ks);
        }
        if (ok) umma_commit(b_qempty + 8 * qs);
      }
      umma_commit(b_done);
      mbar_wait_drain(b_done, 0);
    }
  } else {
    // group g drains key columns [64 g, 64 g + 64) of every key tile; the
    // thread owns query row `row` (TMEM lane) at absolute position pos
    const int g = (warp - 2) >> 2, quarter = warp & 3, row = quarter * 32 + lane;
    const uint32_t lanebase = tmem + ((uint32_t)(quarter * 32) << 16) + g * 64;
    bool live = true;  // after a wait gave up every warp still meets the others at each item's end
    int u = 0, round = 0;
    for (int i = item(0); i < n_items; i = item(++round)) {
    const int h = i % a.hkv, pr0 = item_pr0(i), ntiles = item_tiles(pr0);
    const int pa = p_first + pr0, rows = min(a.p1, a.nq - pr0) * a.G, pos = pa + row / a.G;
    float m = -CUDART_INF_F, l = 0.f;
    for (int it = 0; live && it < ntiles; ++it, ++u) {
      const int as = u & 1;
      if (!warp_wait(b_accfull + 8 * as, (uint32_t)(u >> 1) & 1u, err, abort_flag)) {
        live = false;
        break;
      }
      tc_fence_after();
      float v[64];
      tmem_ld64(lanebase + as * 256, v);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(b_accempty + 8 * as);
      const int key0 = it * 256 + g * 64;
      if (key0 + 63 <= pa) {
        // every row of the tile sees all 64 keys.  The maximum over four
        // independent max3 chains (exact in any order); then exponent
        // arguments, exponentials and sums in three phases with packed
        // fp32x2 operations (each lane of a pair rounds as the scalar op)
        float cm[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) cm[r] = v[r];
#pragma unroll
        for (int i = 4; i < 64; i += 8) {
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (i + 2 * r + 1 < 64) cm[r] = max3(cm[r], v[i + 2 * r], v[i + 2 * r + 1]);
        }
        const float mx = fmaxf(fmaxf(cm[0], cm[1]), fmaxf(cm[2], cm[3]));
        const float mn = fmaxf(m, mx), mnc = mn * c;
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
        for (int i = 0; i < 64; i += 2) fma2(v[i], v[i + 1], c, c, -mnc, -mnc, v[i], v[i + 1]);
#pragma unroll
        for (int i = 0; i < 64; ++i) v[i] = ex2_approx(v[i]);
#pragma unroll
        for (int i = 0; i < 64; i += 4) {
          add2(s0, s1, v[i], v[i + 1]);
          add2(s2, s3, v[i + 2], v[i + 3]);
        }
        l = (m == -CUDART_INF_F ? 0.f : l * ex2_approx((m - mn) * c)) + ((s0 + s1) + (s2 + s3));
        m = mn;
      } else {
        // causal edge: keys key0 + i <= pos only
        const int nv = max(0, min(64, pos - key0 + 1));
        if (nv > 0) {
          float mx = -CUDART_INF_F;
#pragma unroll
          for (int i = 0; i < 64; ++i)
            if (i < nv) mx = fmaxf(mx, v[i]);
          const float mn = fmaxf(m, mx), mnc = mn * c;
          float sacc = 0.f;
#pragma unroll
          for (int i = 0; i < 64; ++i)
            if (i < nv) sacc += ex2_approx(fmaf(v[i], c, -mnc));
          l = (m == -CUDART_INF_F ? 0.f : l * ex2_approx((m - mn) * c)) + sacc;
          m = mn;
        }
      }
    }
    // merge the four groups' states per row in group order (two exchange
    // buffers in turn: one is rewritten after the other's barrier)
    float2* xp = xch + (round & 1) * kPrGroups * 128;
    xp[g * 128 + row] = make_float2(m, l);
    epilogue_sync();
    if (g == 0 && row < rows && live && !*abort_flag) {
      float mm = xp[row].x, ll = xp[row].y;
      for (int o = 1; o < kPrGroups; ++o) {
        const float2 s = xp[o * 128 + row];
        const float mn = fmaxf(mm, s.x);
        if (mn == -CUDART_INF_F) continue;
        const float x = mm == -CUDART_INF_F ? 0.f : ll * exp2f((mm - mn) * c);
        const float y = s.x == -CUDART_INF_F ? 0.f : s.y * exp2f((s.x - mn) * c);
        mm = mn;
        ll = x + y;
      }
      const int prel = pr0 + row / a.G, gq = row - (row / a.G) * a.G;
      const size_t at = ((size_t)h * a.n_ch + prel / a.p2) * a.crp + (size_t)(prel % a.p2) * a.G + gq;
      bias[at] = -mm * c - log2f((float)a.G * ll);
    }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// CLUSTER: a cluster of CTAs per key tile; otherwise one, in code without any
// cluster operations: compiled in, even where a CTA skips them all, they cost
// 0.4 us of a one-chunk CTA's 5 (one row over 50,000 keys, 1,564 such CTAs: the
// column sums 52.9 us, without them 48.8).
template <bool CLUSTER>
__global__ void __maxnreg__(kPrMaxReg)
    k_prompt_colsum(const __grid_constant__ PromptMaps maps, PromptArgs a, const float* bias, float* a_out,
                    uint32_t* err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = pr_align1024(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // a cluster of `split` CTAs per key tile: rank r takes every split-th chunk
  // (keys seen by the most rows first)
  cg::cluster_group cl = cg::this_cluster();
  const int split = CLUSTER ? (int)cl.num_blocks() : 1, rank = CLUSTER ? (int)cl.block_rank() : 0;
  const int unit = blockIdx.x / split, h = unit % a.hkv, kt = unit / a.hkv;
  const int j0 = kt * 128;
  const int p_first = a.n - a.nq;
  const int cstart = (j0 <= p_first ? 0 : (j0 - p_first) / a.p2) + rank;
  const int nitems = cstart < a.n_ch ? (a.n_ch - cstart + split - 1) / split : 0;
  const uint32_t sK = smem_u32(sm + kP2K), sQ = smem_u32(sm + kP2Q);
  float* bias_s = reinterpret_cast<float*>(sm + kP2Bias);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + kP2Bar);
  const uint32_t b_qfull = smem_u32(&bars[0]), b_qempty = smem_u32(&bars[kP2Stages]);
  const uint32_t b_accfull = smem_u32(&bars[2 * kP2Stages]), b_accempty = smem_u32(&bars[2 * kP2Stages + 2]);
  const uint32_t b_k = smem_u32(&bars[2 * kP2Stages + 4]), b_done = smem_u32(&bars[2 * kP2Stages + 5]);
  const uint32_t b_bfull = smem_u32(&bars[2 * kP2Stages + 6]);
  const uint32_t b_bempty = smem_u32(&bars[2 * kP2Stages + 6 + kP2BStages]);
  uint32_t* slot = reinterpret_cast<uint32_t*>(sm + kP2Bar + 8 * (2 * kP2Stages + 6 + 2 * kP2BStages));
  volatile uint32_t* abort_flag = slot + 1;
  float* xch = reinterpret_cast<float*>(sm + kP2Xch);
  float2* sum_s = reinterpret_cast<float2*>(sm + kP2Sum);
  const float c = kPrLog2e * rsqrtf((float)kD);
  const int qrows = a.G * a.p2;  // real lines of a chunk; lines up to 256 stay zero

  // zero the lines of every Q stage that no copy writes, and the bias
  // columns past the copied ones (-inf: they add exact zeros)
  for (int e = threadIdx.x; e < kP2Stages * 2 * (256 - qrows) * 8; e += blockDim.x) {
    const int per_half = (256 - qrows) * 8;
    const int s = e / (2 * per_half), rem = e % (2 * per_half), kb = rem / per_half, w = rem % per_half;
    *reinterpret_cast<uint4*>(sm + kP2Q + s * kP2QStage + kb * 32768 + qrows * 128 + w * 16) = make_uint4(0, 0, 0, 0);
  }
  for (int e = threadIdx.x; e < kP2BStages * 256; e += blockDim.x)
    if ((e & 255) >= a.crp) bias_s[e] = -CUDART_INF_F;
  fence_proxy_async_smem();
  if (threadIdx.x == 0) {
    for (int i = 0; i < kP2Stages; ++i) {
      mbar_init(b_qfull + 8 * i, 1);
      mbar_init(b_qempty + 8 * i, 1);
    }
    // the biases have a ring of their own: the query rows' stage is free as
    // soon as its MMA is done, not when the epilogue has read its biases
    for (int i = 0; i < kP2BStages; ++i) {
      mbar_init(b_bfull + 8 * i, 1);
      mbar_init(b_bempty + 8 * i, 4 * kPrGroups);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(b_accfull + 8 * i, 1);
      mbar_init(b_accempty + 8 * i, 4 * kPrGroups);
    }
    mbar_init(b_k, 1);
    mbar_init(b_done, 1);
    *abort_flag = 0u;
    fence_mbar_init();
    tma_prefetch_desc(&maps.q2);
    tma_prefetch_desc(&maps.k2);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  const float* bias_h = bias + (size_t)h * a.n_ch * a.crp;

  if (warp == 0) {
    if (lane == 0) {
      mbar_arrive_expect_tx(b_k, 32768u);
      tma_load_3d(sK, &maps.k2, b_k, 0, h, j0);
      tma_load_3d(sK + 16384, &maps.k2, b_k, 64, h, j0);
      const uint32_t qbytes = 2u * 128u * (uint32_t)qrows, bbytes = 4u * (uint32_t)a.crp;
      int issued[kP2Stages] = {0, 0}, b_issued[kP2BStages] = {0, 0, 0, 0};
      int ks = 0;
      uint32_t kp = 0u;
      for (int it = 0; it < nitems; ++it, ks = ks + 1 == kP2Stages ? 0 : ks + 1, kp += ks == 0 ? 1u : 0u) {
        if (!mbar_wait(b_qempty + 8 * ks, (kp & 1u) ^ 1u, err, abort_flag)) break;
        const int ch = cstart + it * split, bs = it % kP2BStages;
        mbar_arrive_expect_tx(b_qfull + 8 * ks, qbytes);
        tma_load_3d(sQ + ks * kP2QStage, &maps.q2, b_qfull + 8 * ks, 0, h * a.G, ch * a.p2);
        tma_load_3d(sQ + ks * kP2QStage + 32768, &maps.q2, b_qfull + 8 * ks, 64, h * a.G, ch * a.p2);
        ++issued[ks];
        if (!mbar_wait(b_bempty + 8 * bs, ((uint32_t)(it / kP2BStages) & 1u) ^ 1u, err, abort_flag)) break;
        mbar_arrive_expect_tx(b_bfull + 8 * bs, bbytes);
        bulk_g2s(smem_u32(bias_s + bs * 256), bias_h + (size_t)ch * a.crp, bbytes, b_bfull + 8 * bs);
        ++b_issued[bs];
      }
      if (*abort_flag) {
        mbar_wait_drain(b_k, 0);
        for (int s = 0; s < kP2Stages; ++s)
          if (issued[s]) mbar_wait_drain(b_qfull + 8 * s, (uint32_t)(issued[s] - 1) & 1u);
        for (int s = 0; s < kP2BStages; ++s)
          if (b_issued[s]) mbar_wait_drain(b_bfull + 8 * s, (uint32_t)(b_issued[s] - 1) & 1u);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16(128, 256);
      bool ok = mbar_wait(b_k, 0, err, abort_flag);
      int ks = 0;
      uint32_t kp = 0u;
      for (int it = 0; ok && it < nitems; ++it, ks = ks + 1 == kP2Stages ? 0 : ks + 1, kp += ks == 0 ? 1u : 0u) {
        if (!mbar_wait(b_qfull + 8 * ks, kp & 1u, err, abort_flag)) break;
        const int as = it & 1;
        if (!mbar_wait(b_accempty + 8 * as, ((uint32_t)(it >> 1) & 1u) ^ 1u, err, abort_flag)) break;
        tc_fence_after();
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const uint32_t kb = k >> 2, koff = (k & 3) * 32;
          const uint64_t ad = desc_sw128(sK + kb * 16384 + koff);
          const uint64_t bd = desc_sw128(sQ + ks * kP2QStage + kb * 32768 + koff);
          umma_bf16(tmem + as * 256, ad, bd, idesc, k > 0 ? 1u : 0u);
        }
        umma_commit(b_accfull + 8 * as);
        umma_commit(b_qempty + 8 * ks);
      }
      umma_commit(b_done);
      mbar_wait_drain(b_done, 0);
    }
  } else {
    // group g drains query columns [64 g, 64 g + 64) of every item; the
    // thread owns key j (TMEM lane `row`).  Chunk ch's column col is the row
    // at position p_first + ch P2 + col / G, which attends to j iff
    // col >= (j - chunk's first position) G.
    const int g = (warp - 2) >> 2, quarter = warp & 3, row = quarter * 32 + lane;
    const int j = j0 + row;
    const uint32_t lanebase = tmem + ((uint32_t)(quarter * 32) << 16) + g * 64;
    float sum = 0.f, comp = 0.f;  // compensated running total over the items
    for (int it = 0; it < nitems; ++it) {
      const int as = it & 1, bs = it % kP2BStages;
      if (!warp_wait(b_accfull + 8 * as, (uint32_t)(it >> 1) & 1u, err, abort_flag)) break;
      tc_fence_after();
      float v[64];
      tmem_ld64(lanebase + as * 256, v);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(b_accempty + 8 * as);
      if (!warp_wait(b_bfull + 8 * bs, (uint32_t)(it / kP2BStages) & 1u, err, abort_flag)) break;
      const float4* b4 = reinterpret_cast<const float4*>(bias_s + bs * 256 + g * 64);
      const int p0 = p_first + (cstart + it * split) * a.p2;
      float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
      if (p0 >= j0 + 127) {
        // every row of the chunk sees every key of the tile: exponent
        // arguments, exponentials and sums in three phases, packed fp32x2
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float4 b = b4[i];
          fma2(v[4 * i], v[4 * i + 1], c, c, b.x, b.y, v[4 * i], v[4 * i + 1]);
          fma2(v[4 * i + 2], v[4 * i + 3], c, c, b.z, b.w, v[4 * i + 2], v[4 * i + 3]);
        }
#pragma unroll
        for (int i = 0; i < 64; ++i) v[i] = ex2_approx(v[i]);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          add2(s0, s1, v[4 * i], v[4 * i + 1]);
          add2(s2, s3, v[4 * i + 2], v[4 * i + 3]);
        }
      } else {
        const int colmin = max(0, (j - p0) * a.G) - g * 64;  // first visible column of the group's 64
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float4 b = b4[i];
          s0 += 4 * i >= colmin ? ex2_approx(fmaf(v[4 * i], c, b.x)) : 0.f;
          s1 += 4 * i + 1 >= colmin ? ex2_approx(fmaf(v[4 * i + 1], c, b.y)) : 0.f;
          s2 += 4 * i + 2 >= colmin ? ex2_approx(fmaf(v[4 * i + 2], c, b.z)) : 0.f;
          s3 += 4 * i + 3 >= colmin ? ex2_approx(fmaf(v[4 * i + 3], c, b.w)) : 0.f;
        }
      }
      // this stage's biases are read: count the warp out of it
      __syncwarp();
      if (lane == 0) mbar_arrive(b_bempty + 8 * bs);
      const float y = ((s0 + s1) + (s2 + s3)) - comp;
      const float t = sum + y;
      comp = (t - sum) - y;
      sum = t;
    }
    xch[g * 128 + row] = sum;
    epilogue_sync();
    if (g == 0) {
      float2 total = make_float2(xch[row], 0.f);
      for (int i = 1; i < kPrGroups; ++i) add_exact(total, xch[128 * i + row]);
      sum_s[row] = total;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  // the cluster's sums in rank order, up to 32 groups' and rounded once (after
  // a wait gave up, the keys stay unwritten).  Plain sums of the groups and CTAs
  // put the bases of 300-8,576 positions up to 30 % further from the fp64 result
  // than one CTA's sum of four groups had been; these put them 8-15 % nearer, at
  // 0.9 us of 441 (fp64 additions: the same error, 2.5 us).
  if (CLUSTER) cl.sync();
  if (rank == 0 && threadIdx.x < 128 && j0 + (int)threadIdx.x < a.n) {
    const int j = j0 + threadIdx.x;
    float2 total = sum_s[threadIdx.x];
    bool whole = !*abort_flag;
    if (CLUSTER) {
      for (int r = 1; r < split; ++r) {
        const float2 other = cl.map_shared_rank(sum_s, r)[threadIdx.x];
        add_exact(total, other);
        whole = whole && !*cl.map_shared_rank(slot + 1, r);
      }
    }
    float acc = total.x + total.y;
    if (a.mode == 1) acc /= (float)min(a.nq, a.n - j);
    if (whole) a_out[(size_t)h * a.n + j] = acc;
  }
  if (CLUSTER) cl.sync();  // no CTA leaves while rank 0 may still read its sums
}

// ---- fp32 caches: the same two passes on the CUDA cores --------------------
// Both are products of 64 x 64 tiles (tile.cuh).  1,152 positions of 28 heads:
// row statistics 176 us, column sums 229; with a CTA per query row, each thread
// reading keys from global memory, and one product at a time per thread from
// shared memory they took 2,116 and 2,422.
constexpr int kPrSimtSmem = 2 * kTileFloats * 4;

// Query row r (position r / G of the prompt, head r % G of KV head h's group).
__device__ __forceinline__ const float* prompt_row(const float* q, const PromptArgs& a, int h, int r) {
  const int prel = r / a.G;
  return q + ((size_t)prel * a.hq + h * a.G + (r - prel * a.G)) * kD;
}
// Where its bias lies.
__device__ __forceinline__ size_t prompt_bias_at(const PromptArgs& a, int h, int r) {
  const int prel = r / a.G;
  return ((size_t)h * a.n_ch + prel / a.p2) * a.crp + (size_t)(prel % a.p2) * a.G + (r - prel * a.G);
}

// Pass 1: a cluster of CTAs per (64 query rows, KV head), longest rows first;
// each takes every split-th tile of the keys, and their states are merged in
// rank order.  With one CTA, few rows over a long cache were worked off by a CTA
// or a few: one row of 28 heads over 50,000 keys took 4.05 ms, now 0.60.
template <bool CLUSTER>
__global__ void __launch_bounds__(kTileThreads, kTilesPerSm) k_prompt_rowstats_simt(const float* __restrict__ q,
                                                                                   const float* __restrict__ k,
                                                                                   PromptArgs a, float* bias) {
  extern __shared__ float4 tile_smem[];
  float* qs = reinterpret_cast<float*>(tile_smem);
  float* ks = qs + kTileFloats;
  cg::cluster_group cl = cg::this_cluster();
  const int split = CLUSTER ? (int)cl.num_blocks() : 1, rank = CLUSTER ? (int)cl.block_rank() : 0;
  const int rtile = ((int)gridDim.x - 1 - (int)blockIdx.x) / split;  // a cluster's CTAs follow one another
  const int h = blockIdx.y, r0 = rtile * kTileRows, rows = a.nq * a.G;
  const int nr = min(kTileRows, rows - r0), p_first = a.n - a.nq, ty = tile_ty(), tx = tile_tx();
  const float c = kPrLog2e * rsqrtf((float)kD);
  tile_load(qs, nr, [&](int r) { return prompt_row(q, a, h, r0 + r); });
  float m[kTA], l[kTA];
  int pos[kTA];  // last key of the thread's rows
#pragma unroll
  for (int i = 0; i < kTA; ++i) {
    m[i] = -CUDART_INF_F;
    l[i] = 0.f;
    pos[i] = p_first + (r0 + min(ty + 8 * i, nr - 1)) / a.G;
  }
  const int kend = p_first + (r0 + nr - 1) / a.G + 1;  // keys that some row sees
  for (int j0 = rank * kTileRows; j0 < kend; j0 += split * kTileRows) {
    tile_load(ks, min(kTileRows, kend - j0), [&](int r) { return k + ((size_t)(j0 + r) * a.hkv + h) * kD; });
    tile_ready();
    float d[kTA][kTB];
    tile_dots(qs, ks, d);
#pragma unroll
    for (int i = 0; i < kTA; ++i) {
#pragma unroll
      for (int j = 0; j < kTB; ++j) d[i][j] = j0 + tx + 16 * j <= pos[i] ? d[i][j] * c : -CUDART_INF_F;
      fold_scores(m[i], l[i], d[i]);
    }
    __syncthreads();  // the key tile is rewritten
  }
  merge_rows(m, l, ks);
  float2* states = reinterpret_cast<float2*>(qs);  // (its copies ended in merge_rows, its reads before)
  if (CLUSTER) {
    if (rank > 0 && tx == 0)
#pragma unroll
      for (int i = 0; i < kTA; ++i) states[ty + 8 * i] = make_float2(m[i], l[i]);
    cl.sync();
  }
  if (rank == 0 && tx == 0)
#pragma unroll
    for (int i = 0; i < kTA; ++i) {
      const int r = ty + 8 * i;
      if (CLUSTER) {  // every scaling is by a power of two (fold_scores), and the sum is rounded once
        float mx = m[i];
        for (int o = 1; o < split; ++o) mx = fmaxf(mx, cl.map_shared_rank(states, o)[r].x);
        auto scaled = [&](float m2, float l2) { return l2 == 0.f || m2 == mx ? l2 : l2 * exp2f(m2 - mx); };
        float2 total = make_float2(scaled(m[i], l[i]), 0.f);
        for (int o = 1; o < split; ++o) {
          const float2 s = cl.map_shared_rank(states, o)[r];
          add_exact(total, scaled(s.x, s.y));
        }
        m[i] = mx;
        l[i] = total.x + total.y;
      }
      if (r < nr) bias[prompt_bias_at(a, h, r0 + r)] = -m[i] - log2f((float)a.G * l[i]);
    }
  if (CLUSTER) cl.sync();  // no CTA leaves while rank 0 may still read its states
}

// Pass 2: a cluster of CTAs per (64 keys, KV head), each taking every split-th
// tile of the query rows that can see the keys; their sums are added in rank
// order.
__global__ void __launch_bounds__(kTileThreads, kTilesPerSm) k_prompt_colsum_simt(const float* __restrict__ q,
                                                                                 const float* __restrict__ k,
                                                                                 PromptArgs a, const float* bias,
                                                                                 float* a_out) {
  extern __shared__ float4 tile_smem[];
  float* ks = reinterpret_cast<float*>(tile_smem);
  float* qs = ks + kTileFloats;
  cg::cluster_group cl = cg::this_cluster();
  const int split = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int h = blockIdx.y, j0 = (int)blockIdx.x / split * kTileRows, rows = a.nq * a.G;
  const int p_first = a.n - a.nq, ty = tile_ty(), tx = tile_tx();
  const float c = kPrLog2e * rsqrtf((float)kD);
  const int r_start = j0 <= p_first ? 0 : (j0 - p_first) * a.G;  // rows before it see no key of the tile
  tile_load(ks, min(kTileRows, a.n - j0), [&](int r) { return k + ((size_t)(j0 + r) * a.hkv + h) * kD; });
  float2 acc[kTA];
#pragma unroll
  for (int i = 0; i < kTA; ++i) acc[i] = make_float2(0.f, 0.f);
  for (int rt = r_start + rank * kTileRows; rt < rows; rt += split * kTileRows) {
    const int nr = min(kTileRows, rows - rt);
    tile_load(qs, nr, [&](int r) { return prompt_row(q, a, h, rt + r); });
    float bs[kTB];
    int pos[kTB];  // last key of the thread's rows; -1: no row
#pragma unroll
    for (int j = 0; j < kTB; ++j) {
      const int r = tx + 16 * j;
      bs[j] = r < nr ? __ldg(bias + prompt_bias_at(a, h, rt + r)) : 0.f;
      pos[j] = r < nr ? p_first + (rt + r) / a.G : -1;
    }
    tile_ready();
    float d[kTA][kTB];
    tile_dots(ks, qs, d);
#pragma unroll
    for (int i = 0; i < kTA; ++i) {
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < kTB; ++j) sum += j0 + ty + 8 * i <= pos[j] ? exp2f(fmaf(d[i][j], c, bs[j])) : 0.f;
      add_exact(acc[i], sum);
    }
    __syncthreads();  // the query tile is rewritten
  }
  float2* sums = reinterpret_cast<float2*>(qs);
  sum_rows(acc, sums);
  if (split > 1)
    cl.sync();
  else
    __syncthreads();
  const int j = j0 + threadIdx.x;
  if (rank == 0 && threadIdx.x < kTileRows && j < a.n) {
    float2 total = sums[threadIdx.x];
    for (int r = 1; r < split; ++r) add_exact(total, cl.map_shared_rank(sums, r)[threadIdx.x]);
    float sum = total.x + total.y;
    if (a.mode == 1) sum /= (float)min(a.nq, a.n - j);
    a_out[(size_t)h * a.n + j] = sum;
  }
  if (split > 1) cl.sync();  // no CTA leaves while rank 0 may still read its sums
}

// ---- host --------------------------------------------------------------

namespace {

PFN_cuTensorMapEncodeTiled_v12000 prompt_encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &qr) ==
            cudaSuccess &&
        qr == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
  }
  return fn;
}

// q [nq][hq][128] bf16 as a 3-D tensor (d, query head, position); box 64 x
// G x P with the 128-byte swizzle; positions past nq read as zero.
cudaError_t make_prompt_qmap(CUtensorMap* m, const void* q, int nq, int hq, int G, int P) {
  auto fn = prompt_encode_fn();
  if (!fn) return cudaErrorNotSupported;
  cuuint64_t dims[3] = {(cuuint64_t)kD, (cuuint64_t)hq, (cuuint64_t)nq};
  cuuint64_t strides[2] = {(cuuint64_t)kD * 2, (cuuint64_t)hq * kD * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)G, (cuuint32_t)P};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(q), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

PromptArgs prompt_args(int n, int nq, int hq, int hkv, int mode) {
  PromptArgs a;
  a.n = n;
  a.nq = nq;
  a.hq = hq;
  a.hkv = hkv;
  a.G = hq / hkv;
  a.p1 = 128 / a.G;
  a.p2 = 256 / a.G;
  a.n_mt = (nq + a.p1 - 1) / a.p1;
  a.n_ch = (nq + a.p2 - 1) / a.p2;
  a.crp = (a.G * a.p2 + 3) / 4 * 4;
  a.mode = mode;
  return a;
}

}  // namespace

// CTAs per key tile of pass 2.  A tile's chunks cannot be shared between
// waves, so the pass ends with the CTA of the most chunks (the first keys'
// tiles: every chunk) or, with many tiles, when the SMs have worked off all of
// them: about total / SMs + longest / 2 chunks, plus 6 per CTA an SM runs.  It
// fixes how the sums are grouped, so it depends on the shape alone (152 SMs).
static int prompt_split(const PromptArgs& a) {
  constexpr int nsm = 152;
  const long long tiles = (a.n + 127) / 128;
  long long chunks = 0;
  for (long long t = 0; t < tiles; ++t) {
    const long long j0 = t * 128, pf = a.n - a.nq;
    chunks += a.n_ch - (j0 <= pf ? 0 : (j0 - pf) / a.p2);
  }
  int best = 1;
  double best_cost = 0.0;
  for (int s = 1; s <= kP2MaxSplit && s <= std::max(1, a.n_ch); s <<= 1) {
    const double ctas = (double)tiles * a.hkv * s, longest = (double)a.n_ch / s;
    const double cost = std::max((double)chunks * a.hkv / nsm + longest / 2, longest) + 6.0 * std::ceil(ctas / nsm);
    if (s == 1 || cost < best_cost) {
      best = s;
      best_cost = cost;
    }
  }
  return best;
}

size_t prompt_bias_bytes(int n, int nq, int hq, int hkv) {
  const PromptArgs a = prompt_args(n, nq, hq, hkv, 0);
  return (size_t)hkv * a.n_ch * a.crp * 4;
}

cudaError_t launch_prompt_score(DType dt, const void* q, const void* k, int n, int nq, int hq, int hkv, int mode,
                                float* a_out, float* bias, uint32_t* err, cudaStream_t st) {
  const PromptArgs a = prompt_args(n, nq, hq, hkv, mode);
  if (a.p1 < 1) return cudaErrorNotSupported;
  if (dt == kF32) {
    cudaError_t e;
    const float* qf = static_cast<const float*>(q);
    const float* kf = static_cast<const float*>(k);
    const int rows = nq * a.G, ktiles = (n + kTileRows - 1) / kTileRows, rtiles = (rows + kTileRows - 1) / kTileRows;
    if ((e = cudaFuncSetAttribute(k_prompt_rowstats_simt<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  kPrSimtSmem)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(k_prompt_rowstats_simt<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  kPrSimtSmem)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(k_prompt_colsum_simt, cudaFuncAttributeMaxDynamicSharedMemorySize, kPrSimtSmem)) !=
            cudaSuccess)
      return e;
    // The largest cluster of 1, 2, 4 or 8 CTAs per tile, at most `others`, that
    // keeps the grid within `limit` CTAs.  It fixes how the sums are grouped, so
    // it depends on the shape alone.
    auto clusters = [&](long long tiles, int others, int limit) {
      int s = 1;
      while (2 * s <= others && 2 * s <= kP2MaxSplit && tiles * hkv * 2 * s <= limit) s *= 2;
      return s;
    };
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.blockDim = dim3(kTileThreads);
    cfg.dynamicSmemBytes = kPrSimtSmem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    auto grid = [&](int tiles, int split) {
      cfg.gridDim = dim3((unsigned)(tiles * split), hkv);
      attr[0].val.clusterDim.x = (unsigned)split;
      cfg.numAttrs = split > 1 ? 1 : 0;
    };
    {
      TimingScope ts("prompt_rowstats_simt", st);
      // Clusters while they fill the SMs' places once, with three key tiles or
      // more for each CTA: with one or two it spends what it spares on its copy
      // of the query tile and on the merge (300 keys, 1,561 rows: 37 us, in
      // clusters of two 40; 900 keys, one row: 86, in clusters of four 39).
      const int split = clusters(rtiles, ktiles / 3, 152 * kTilesPerSm);
      grid(rtiles, split);
      e = cudaLaunchKernelEx(&cfg, split > 1 ? k_prompt_rowstats_simt<true> : k_prompt_rowstats_simt<false>, qf, kf, a,
                             bias);
    }
    if (e != cudaSuccess || (e = cudaGetLastError()) != cudaSuccess) return e;
    TimingScope ts("prompt_colsum_simt", st);
    // until the CTAs fill the SMs four times (the first tiles see every row, the last ones few)
    grid(ktiles, clusters(ktiles, rtiles, 4 * 152 * kTilesPerSm));
    e = cudaLaunchKernelEx(&cfg, k_prompt_colsum_simt, qf, kf, a, (const float*)bias, a_out);
    return e != cudaSuccess ? e : cudaGetLastError();
  }
  PromptMaps maps;
  cudaError_t e = make_prompt_qmap(&maps.q1, q, nq, hq, a.G, a.p1);
  if (e == cudaSuccess) e = make_prompt_qmap(&maps.q2, q, nq, hq, a.G, a.p2);
  if (e == cudaSuccess) e = make_row_map(&maps.k1, k, n, hkv, 256);
  if (e == cudaSuccess) e = make_row_map(&maps.k2, k, n, hkv, 128);
  if (e != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_prompt_rowstats, cudaFuncAttributeMaxDynamicSharedMemorySize, kP1Smem)) !=
      cudaSuccess)
    return e;
  const int split = prompt_split(a);
  auto cs_kernel = split > 1 ? k_prompt_colsum<true> : k_prompt_colsum<false>;
  if ((e = cudaFuncSetAttribute(cs_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kP2Smem)) != cudaSuccess)
    return e;
  int nsm = 0, dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  {
    TimingScope ts("prompt_rowstats", st);
    k_prompt_rowstats<<<(unsigned)std::min(nsm, a.n_mt * hkv), kPrThreads, kP1Smem, st>>>(maps, a, bias, err);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3((unsigned)((n + 127) / 128 * hkv * split));
  cfg.blockDim = dim3(kPrThreads);
  cfg.dynamicSmemBytes = kP2Smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)split;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = split > 1 ? 1 : 0;
  TimingScope ts("prompt_colsum", st);
  if ((e = cudaLaunchKernelEx(&cfg, cs_kernel, maps, a, (const float*)bias, a_out, err)) != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace stl
