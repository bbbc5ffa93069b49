// Selection kernel.  One cluster of CL CTAs per (layer, KV head); CTA c of a
// cluster owns the contiguous token range [c*chunk, (c+1)*chunk) and keeps
// its keys in shared memory for every pass.
//   kSelGate: rho_i = |k_i|^-1 * TSG's row maximum (Eq. 6), tau =
//             the min(B, |pool|)-th smallest rho (Eq. 7), gate = rho <= tau
//             (Eq. 8).
//   kSelTopk: S from Eq. 9, then the B-th largest S and an ordered stream
//             compaction that emits the kept indices in ascending order,
//             equal scores resolved towards lower indices.
// Both selections are exact selects on the order-preserving uint32 images of
// the fp32 values (cluster_select below): the cluster's key range, a 1,024-bin
// histogram of it, and the few keys of the chosen bin gathered into every CTA
// and resolved there.
#include <cooperative_groups.h>

#include <algorithm>

#include "fit_cache.h"
#include "kernels.cuh"

namespace cg = cooperative_groups;

namespace stl {

constexpr int kSelThreads = 512;  // two bins of a histogram pass each
constexpr int kSelMaxCluster = 8;
constexpr int kSelMaxChunk = 49152;  // keys per CTA held in shared memory (192 KB)

constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelBins = 1024;           // bins of a histogram pass: two per thread
constexpr int kSelGather = 2 * kSelThreads;  // most keys a chosen bin may hold to be gathered
static_assert(kSelBins == 2 * kSelThreads, "a thread sums two bins");
static_assert(kSelMaxChunk < 65536, "a CTA's bins and counts are 16-bit");

// The keys above a pivot (see cluster_select), of a thread, a CTA or the cluster.
struct SelStats {
  uint32_t n, mn, mx;  // their count, the smallest and the largest
};

struct SelShared {
  uint32_t hist[2][kSelBins / 2];  // bins 2t (low half) and 2t + 1 of this CTA's keys, by pass parity
  uint32_t cand[kSelGather];       // the cluster's keys of the chosen bin
  uint32_t fine[3][256];           // histograms of them
  SelStats stats[2][2];   // of this CTA: per select of the kernel, above the pivot; at and below it
  uint32_t n_list;        // keys of the CTA in the chosen bin
  uint32_t dig[4];        // (bin, count above it, count in it, count in it of the CTAs before this one)
  uint32_t warp_tot[32];
  uint32_t counts[2];     // (greater, equal) of this CTA for the compaction
  float warp_max[32];
  float cta_max;          // read by the cluster's other CTAs
  int32_t fr_off[kMaxFrames + 1];  // first token of every frame; fr_off[F] = INT_MAX
  int32_t fr_vend[kMaxFrames];     // end of every frame's visual span
};

// Cluster barrier (a block barrier when the CTA is alone).
__device__ __forceinline__ void cluster_barrier(cg::cluster_group& cl, int ncta) {
  if (ncta > 1)
    cl.sync();
  else
    __syncthreads();
}

// Maximum of v over every thread of the cluster (every CTA must call it).
__device__ float cluster_max(cg::cluster_group& cl, float v, SelShared& sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if (lane == 0) sh.warp_max[wid] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    float m = sh.warp_max[0];
    for (int w = 1; w < nw; ++w) m = fmaxf(m, sh.warp_max[w]);
    sh.cta_max = m;
  }
  cluster_barrier(cl, (int)cl.num_blocks());
  float m = -CUDART_INF_F;
  for (int r = 0; r < (int)cl.num_blocks(); ++r) m = fmaxf(m, *cl.map_shared_rank(&sh.cta_max, r));
  return m;
}

// Exclusive block-wide prefix sum of v; *total receives the block sum.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* warp_tot,
                                                         uint32_t* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[wid] = x;
  __syncthreads();
  if (wid == 0) {
    uint32_t t = lane < nw ? warp_tot[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    warp_tot[lane] = t;
  }
  __syncthreads();
  const uint32_t before = wid ? warp_tot[wid - 1] : 0u;
  *total = warp_tot[nw - 1];
  __syncthreads();
  return before + x - v;
}

__device__ __forceinline__ void stats_init(SelStats& st) { st = {0u, 0xffffffffu, 0u}; }
__device__ __forceinline__ void stats_add(SelStats& st, uint32_t key, uint32_t pivot) {
  if (key > pivot) {
    ++st.n;
    st.mn = min(st.mn, key);
    st.mx = max(st.mx, key);
  }
}
__device__ __forceinline__ void stats_reduce(SelStats& st) {  // over the warp
  st.n = __reduce_add_sync(0xffffffffu, st.n);
  st.mn = __reduce_min_sync(0xffffffffu, st.mn);
  st.mx = __reduce_max_sync(0xffffffffu, st.mx);
}
// The cluster's statistics from every thread's (`cta` initialised before).
__device__ __forceinline__ SelStats stats_cluster(cg::cluster_group& cl, int ncta, SelStats st, SelStats* cta) {
  const int lane = threadIdx.x & 31;
  stats_reduce(st);
  if (lane == 0) {
    atomicAdd(&cta->n, st.n);
    atomicMin(&cta->mn, st.mn);
    atomicMax(&cta->mx, st.mx);
  }
  cluster_barrier(cl, ncta);
  stats_init(st);
  if (lane < ncta) st = *cl.map_shared_rank(cta, lane);
  stats_reduce(st);
  return st;
}

struct Selected {
  uint32_t T, need;  // the top k: every key > T, and `need` of the keys == T
};

// The k largest of the cluster's keys.  `mine`: this thread's statistics of
// the keys above `pivot`, a value that many keys may share (0 for a closed
// gate's score, or the mark of an empty slot): keys equal to it are counted
// there instead of piling up in one bin.  set_only: the caller needs the set,
// not the k-th key itself, so a bin that holds exactly the keys still needed
// ends the select (T = its lower bound - 1, need = 0).  `sel` numbers the
// kernel's selects, `pass` its histogram passes.
//
// The range [lo, hi] of the keys that can hold the k-th is known after one
// exchange of the CTAs' statistics; a pass cuts it into 1,024 equal bins,
// sums them over the cluster (a thread sums two bins, packed 16-bit in the
// CTAs' copies) and finds the k-th key's bin.  If that bin's keys are few,
// every CTA sends its own to all the others, and each resolves them alone;
// else the bin becomes the range of the next pass (at most four: 32 bits).
// That is three cluster barriers for an ordinary distribution, each of which
// costs 0.6 us in a cluster of 4 and 1.2 us in one of 16.  Not inlined: the
// kernel's second select then finds its instructions in the SM's cache, which
// is worth 3 us of the 9-12 that a cold one takes.
//
// What the cluster's other CTAs read or write is reused only after a later
// barrier that follows every such access: a pass's bins two passes later, the
// gathered keys in the next select.
__device__ __noinline__ Selected cluster_select(int ncta, const uint32_t* keys, int len, uint32_t k, uint32_t pivot,
                                                SelStats mine, SelShared& sh, int sel, int& pass, bool set_only) {
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int rank = (int)cl.block_rank();
  sh.hist[pass & 1][tid] = 0u;
  if (tid == 0) sh.n_list = 0u;
  SelStats st = stats_cluster(cl, ncta, mine, &sh.stats[sel][0]);  // (the keys are written, too)
  uint32_t need = k;
  if (need > st.n) {
    // the k-th is the pivot or below: its count and the range below it
    need -= st.n;
    stats_init(mine);
    uint32_t n_eq = 0;
    for (int i = tid; i < len; i += kSelThreads) {
      const uint32_t key = keys[i];
      n_eq += key == pivot;
      if (key < pivot) {
        mine.mn = min(mine.mn, key);
        mine.mx = max(mine.mx, key);
      }
    }
    mine.n = n_eq;
    st = stats_cluster(cl, ncta, mine, &sh.stats[sel][1]);
    if (need <= st.n) return {pivot, need};
    need -= st.n;
  }
  uint32_t lo = st.mn, hi = st.mx;
  for (int it = 0; it < 4; ++it) {  // a pass leaves at most a 1,024th of the range: four are enough for 32 bits
    if (lo == hi) break;  // equal keys
    const uint32_t span = hi - lo;
    const int shift = max(0, 22 - __clz(span));  // span >> shift < 1,024
    uint32_t* hist = sh.hist[pass & 1];
    ++pass;
    if (it > 0) {
      hist[tid] = 0u;
      __syncthreads();
    }
    auto count = [&](uint32_t r, uint32_t n) {  // n keys of r's bin, r = key - lo
      const uint32_t b = r >> shift;
      if (r <= span) atomicAdd(&hist[b >> 1], b & 1u ? n << 16 : n);
    };
    // Four neighbouring keys of one bin are added at once: where most keys
    // crowd into a bin, their additions wait for one another (one layer with
    // near-duplicate frames, 4 x 53,600 tokens: 36 -> 35 us; 112 x 53,600 scores,
    // most within 0.1 % of one another and a few far off: 69 -> 58).
    for (int i = tid; i < len >> 2; i += kSelThreads) {
      const uint4 x = reinterpret_cast<const uint4*>(keys)[i];
      const uint32_t r0 = x.x - lo, r1 = x.y - lo, r2 = x.z - lo, r3 = x.w - lo;
      if (max(max(r0, r1), max(r2, r3)) <= span && ((r0 ^ r1) | (r0 ^ r2) | (r0 ^ r3)) >> shift == 0u) {
        count(r0, 4u);
      } else {
        count(r0, 1u);
        count(r1, 1u);
        count(r2, 1u);
        count(r3, 1u);
      }
    }
    if (tid < (len & 3)) count(keys[(len & ~3) + tid] - lo, 1u);
    cluster_barrier(cl, ncta);
    uint32_t c0 = 0, c1 = 0, b0 = 0, b1 = 0;  // counts of the thread's bins; of the CTAs before this one
    for (int r0 = 0; r0 < ncta; r0 += 8) {    // eight remote reads in flight
      uint32_t v[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) v[r] = r0 + r < ncta ? cl.map_shared_rank(hist, r0 + r)[tid] : 0u;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        c0 += v[r] & 0xffffu;
        c1 += v[r] >> 16;
        if (r0 + r < rank) {
          b0 += v[r] & 0xffffu;
          b1 += v[r] >> 16;
        }
      }
    }
    // keys in the bins above the thread's two: in its warp, then in the warps above
    uint32_t incl = c0 + c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_down_sync(0xffffffffu, incl, o);
      if (lane + o < 32) incl += v;
    }
    if (lane == 0) sh.warp_tot[wid] = incl;
    __syncthreads();
    const uint32_t over = __reduce_add_sync(0xffffffffu, lane > wid && lane < kSelWarps ? sh.warp_tot[lane] : 0u);
    const uint32_t above = over + incl - c0 - c1;
    if (above < need && need <= above + c0 + c1) {
      const bool up = need <= above + c1;
      sh.dig[0] = 2 * tid + (up ? 1 : 0);
      sh.dig[1] = up ? above : above + c1;
      sh.dig[2] = up ? c1 : c0;
      sh.dig[3] = up ? b1 : b0;
    }
    __syncthreads();
    const uint32_t in_bin = sh.dig[2], first = sh.dig[3];
    need -= sh.dig[1];
    lo += sh.dig[0] << shift;
    if (shift == 0) break;
    if (set_only && in_bin == need && lo != 0u) return {lo - 1u, 0u};
    hi = lo + min(hi - lo, (1u << shift) - 1u);
    if (in_bin > kSelGather) continue;
    // list the bin's keys, then send the list to every CTA
    const uint32_t width = hi - lo;
    auto list = [&](uint32_t key) {
      if (key - lo <= width) sh.cand[first + atomicAdd(&sh.n_list, 1u)] = key;
    };
    for (int i = tid; i < len >> 2; i += kSelThreads) {
      const uint4 x = reinterpret_cast<const uint4*>(keys)[i];
      list(x.x);
      list(x.y);
      list(x.z);
      list(x.w);
    }
    if (tid < (len & 3)) list(keys[(len & ~3) + tid]);
    if (tid < 256) sh.fine[0][tid] = 0u;
    __syncthreads();
    if (ncta > 1) {
      const uint32_t n = sh.n_list;
      for (uint32_t i = tid; i < n; i += kSelThreads) {
        const uint32_t key = sh.cand[first + i];
        for (int r = 0; r < ncta; ++r)
          if (r != rank) cl.map_shared_rank(sh.cand, r)[first + i] = key;
      }
      cl.sync();
    }
    if (in_bin <= 32) {
      // every warp alone, a key per lane: the k-th has `need` keys at or
      // above it and fewer than that above
      const uint32_t key = lane < in_bin ? sh.cand[lane] : 0u;
      uint32_t gt = 0, ge = 0;
      for (uint32_t x = 0; x < in_bin; ++x) {
        const uint32_t o = __shfl_sync(0xffffffffu, key, x);
        gt += o > key;
        ge += o >= key;
      }
      const bool is = lane < in_bin && gt < need && need <= ge;
      const int src = __ffs(__ballot_sync(0xffffffffu, is)) - 1;
      lo = __shfl_sync(0xffffffffu, key, src);
      need -= __shfl_sync(0xffffffffu, gt, src);
      break;
    }
    // 256 equal bins of the range at a time (it is below 2^22), every warp
    // finding the bin for itself; three histograms in turn, so that the one
    // zeroed for the next round is not the one read last
    const uint32_t k0 = tid < in_bin ? sh.cand[tid] : 0u;  // below lo: not counted
    const uint32_t k1 = tid + kSelThreads < in_bin ? sh.cand[tid + kSelThreads] : 0u;
    for (int round = 0; round < 3 && lo != hi; ++round) {
      const uint32_t w = hi - lo;
      const int s = max(0, 24 - __clz(w));  // w >> s < 256
      uint32_t* h = sh.fine[round];
      if (tid < in_bin && k0 - lo <= w) atomicAdd(&h[(k0 - lo) >> s], 1u);
      if (tid + kSelThreads < in_bin && k1 - lo <= w) atomicAdd(&h[(k1 - lo) >> s], 1u);
      if (round < 2 && tid < 256) h[256 + tid] = 0u;
      __syncthreads();
      uint32_t c[8], sum = 0;
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        c[b] = h[lane * 8 + b];
        sum += c[b];
      }
      uint32_t in = sum;  // over this lane and the ones above
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_down_sync(0xffffffffu, in, o);
        if (lane + o < 32) in += v;
      }
      uint32_t up = in - sum, bin = 0, cnt = 0, left = 0;
      const bool here = up < need && need <= in;
#pragma unroll
      for (int b = 7; b >= 0; --b) {
        if (up < need && need <= up + c[b]) {
          bin = lane * 8 + b;
          cnt = c[b];
          left = need - up;
        }
        up += c[b];
      }
      const int src = __ffs(__ballot_sync(0xffffffffu, here)) - 1;
      bin = __shfl_sync(0xffffffffu, bin, src);
      cnt = __shfl_sync(0xffffffffu, cnt, src);
      need = __shfl_sync(0xffffffffu, left, src);
      lo += bin << s;
      if (s == 0) break;
      if (set_only && cnt == need && lo != 0u) return {lo - 1u, 0u};
      hi = lo + min(hi - lo, (1u << s) - 1u);
    }
    break;
  }
  return {lo, need};
}

// Warms L2 with the 128-byte lines of x[j0, j1) (one prefetch per line):
// the token loops then find their inputs in L2 instead of waiting on DRAM
// once per batch.
__device__ __forceinline__ void prefetch_l2(const void* x, size_t elem, int j0, int j1) {
  const char* b = static_cast<const char*>(x);
  const size_t lo = (size_t)j0 * elem, hi = (size_t)j1 * elem;
  for (size_t o = (lo & ~(size_t)127) + (size_t)threadIdx.x * 128; o < hi; o += (size_t)blockDim.x * 128)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(b + o));
}

// Token kinds of the flat loops.
constexpr int kTokText = 0;  // not inside any frame's visual span
constexpr int kTokPool = 1;  // visual token of a historical frame (the TSG pool)
constexpr int kTokCur = 2;   // visual token of the current (last) frame

// Last frame starting at or before token t (-1: none), on the shared copy
// of the frame table.
__device__ __forceinline__ int frame_at(const SelShared& sh, int F, int t) {
  int lo = 0, hi = F - 1, f = -1;
  while (lo <= hi) {
    const int mid = (lo + hi) >> 1;
    if (sh.fr_off[mid] <= t) {
      f = mid;
      lo = mid + 1;
    } else {
      hi = mid - 1;
    }
  }
  return f;
}

// Visits the tokens j0 + threadIdx.x + k * blockDim.x of [j0, j1) in
// batches of U per thread: load(t, kind) runs for the whole batch before
// use(t, kind, value) runs for any of it, so the batch's memory latencies
// overlap.  Each thread tracks the frame of its (increasing) tokens in the
// shared copy of the frame table (fr_off ends with INT_MAX).
template <int U, class Load, class Use>
__device__ __forceinline__ void for_tokens(const SelShared& sh, int F, int j0, int j1, Load load, Use use) {
  const int B = blockDim.x;
  int f = frame_at(sh, F, j0 + (int)threadIdx.x);
  for (int base = j0 + (int)threadIdx.x; base < j1; base += U * B) {
    int kind[U];
    decltype(load(0, 0)) v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int t = base + u * B;
      kind[u] = -1;
      if (t < j1) {
        while (sh.fr_off[f + 1] <= t) ++f;
        const bool vis = f >= 0 && t < sh.fr_vend[f];
        kind[u] = vis ? (f + 1 < F ? kTokPool : kTokCur) : kTokText;
        v[u] = load(t, kind[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (kind[u] >= 0) use(base + u * B, kind[u], v[u]);
  }
}

// The same visit in groups of four consecutive tokens t0 .. t0 + 3 (t0 =
// j0 + 4 (tid + k B)), for 128-bit loads and stores: j0, j1 and every row
// base are multiples of four tokens.  kinds[e] is the kind of t0 + e (one
// comparison for a group inside one visual span or text run).
template <class Load4, class Use4>
__device__ __forceinline__ void for_tokens4(const SelShared& sh, int F, int j0, int j1, Load4 load4, Use4 use4) {
  const int B = blockDim.x;
  int f = frame_at(sh, F, j0 + 4 * (int)threadIdx.x);
  for (int t0 = j0 + 4 * (int)threadIdx.x; t0 < j1; t0 += 4 * B) {
    int kinds[4];
    while (sh.fr_off[f + 1] <= t0) ++f;
    const int vend = f >= 0 ? sh.fr_vend[f] : -1, next = sh.fr_off[f + 1];
    if (t0 + 3 < vend || (t0 >= vend && t0 + 3 < next)) {  // one kind for the group
      const int k = t0 < vend ? (f + 1 < F ? kTokPool : kTokCur) : kTokText;
#pragma unroll
      for (int e = 0; e < 4; ++e) kinds[e] = k;
    } else {  // the group straddles a span or frame boundary
      int fe = f;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int t = t0 + e;
        while (sh.fr_off[fe + 1] <= t) ++fe;
        kinds[e] = fe >= 0 && t < sh.fr_vend[fe] ? (fe + 1 < F ? kTokPool : kTokCur) : kTokText;
      }
    }
    const auto v = load4(t0, kinds);
    use4(t0, kinds, v);
  }
}

struct RhoIn4 {
  uint4 m;
  float4 rn;
};
struct ScoreIn4 {
  float4 A, P;
  uint32_t G;  // four gate bytes
};

__global__ void __launch_bounds__(kSelThreads, 4) k_select(Problem p, const __grid_constant__ FrameTable ft,
                                                        SelectArgs a) {
  extern __shared__ uint4 key_smem[];  // its type aligns it: cluster_select reads four keys at a time
  uint32_t* const keys = reinterpret_cast<uint32_t*>(key_smem);
  __shared__ SelShared sh;
  cg::cluster_group cl = cg::this_cluster();
  const int ncta = (int)cl.num_blocks(), c = (int)cl.block_rank();
  const int l = blockIdx.y / p.hkv, h = blockIdx.y % p.hkv, n = p.n, tid = threadIdx.x;
  pdl_trigger();
  const int chunk = ((n + ncta - 1) / ncta + 3) & ~3;  // four-token groups never straddle two CTAs
  const int j0 = min(n, c * chunk), j1 = min(n, j0 + chunk), len = j1 - j0;
  const bool vec = (n & 3) == 0;  // every row base [Hkv][N] is 16-byte aligned
  const size_t hn = (size_t)h * n;
  const int F = ft.n_frames;
  int pass = 0;
  int pool = 0;
  for (int f = 0; f + 1 < F; ++f) pool += ft.gh[f] * ft.gw[f];
  // the frame table in shared memory for the token loops' frame tracking
  for (int f = tid; f <= F; f += blockDim.x) {
    sh.fr_off[f] = f < F ? ft.off[f] : 0x7fffffff;
    if (f < F) sh.fr_vend[f] = ft.off[f] + ft.gh[f] * ft.gw[f];
  }
  if (tid < 4) stats_init(sh.stats[tid >> 1][tid & 1]);
  __syncthreads();
  // tau comes from a selection only when there is a pool and TSG is on;
  // otherwise tau = NaN and every gate stays open
  const bool gate_sel = (a.mode & kSelGate) && pool > 0 && a.tsg_enable;
  float tau = CUDART_NAN_F;
  uint32_t kt_gate = 0u;  // gate: rho <= tau, i.e. key (~float_key(rho)) >= kt_gate
  uint8_t* gate = a.gate.base ? a.gate.at(l) + hn : nullptr;

  SelStats ks;  // of the keys this thread writes
  if (a.mode & kSelGate) {
    stats_init(ks);
    float* rho = a.rho.at(l) + hn;
    const uint32_t* rk = a.rho_key.at(l) + hn;
    const float* rn = a.rn.at(l) + hn;
    prefetch_l2(rk, 4, j0, j1);
    prefetch_l2(rn, 4, j0, j1);
    // rho of every token: pool tokens from TSG's maxima and 1/|k_i|, NaN
    // elsewhere; the selection keys are complements (m-th smallest rho ==
    // m-th largest key), 0 marks a token outside the pool.  Finish Eq. 6
    // with the row's own term: times 1/|k_i| (cosine), nothing (dot), minus
    // |k_i|^2 (negative squared L2).
    auto finish = [&](uint32_t key, float rnv) {
      const float m = key_float(key);
      return a.tsg_metric == kTsgCosine ? m * rnv : (a.tsg_metric == kTsgDot ? m : m - 1.f / (rnv * rnv));
    };
    if (vec) {
      for_tokens4(
          sh, F, j0, j1,
          [&](int t0, const int (&kinds)[4]) {
            RhoIn4 r;
            r.m = make_uint4(0u, 0u, 0u, 0u);
            r.rn = make_float4(0.f, 0.f, 0.f, 0.f);
            if (kinds[0] == kTokPool || kinds[1] == kTokPool || kinds[2] == kTokPool || kinds[3] == kTokPool) {
              r.m = __ldg(reinterpret_cast<const uint4*>(rk + t0));
              r.rn = __ldg(reinterpret_cast<const float4*>(rn + t0));
            }
            return r;
          },
          [&](int t0, const int (&kinds)[4], const RhoIn4& v) {
            const float r0 = kinds[0] == kTokPool ? finish(v.m.x, v.rn.x) : CUDART_NAN_F;
            const float r1 = kinds[1] == kTokPool ? finish(v.m.y, v.rn.y) : CUDART_NAN_F;
            const float r2 = kinds[2] == kTokPool ? finish(v.m.z, v.rn.z) : CUDART_NAN_F;
            const float r3 = kinds[3] == kTokPool ? finish(v.m.w, v.rn.w) : CUDART_NAN_F;
            if (a.write_stages) *reinterpret_cast<float4*>(rho + t0) = make_float4(r0, r1, r2, r3);
            const uint4 kv = make_uint4(kinds[0] == kTokPool ? ~float_key(r0) : 0u,
                                        kinds[1] == kTokPool ? ~float_key(r1) : 0u,
                                        kinds[2] == kTokPool ? ~float_key(r2) : 0u,
                                        kinds[3] == kTokPool ? ~float_key(r3) : 0u);
            *reinterpret_cast<uint4*>(keys + (t0 - j0)) = kv;
            stats_add(ks, kv.x, 0u);
            stats_add(ks, kv.y, 0u);
            stats_add(ks, kv.z, 0u);
            stats_add(ks, kv.w, 0u);
          });
    } else
    for_tokens<2>(
        sh, F, j0, j1,
        [&](int t, int kind) {
          return kind == kTokPool ? make_uint2(__ldg(rk + t), __float_as_uint(__ldg(rn + t))) : make_uint2(0u, 0u);
        },
        [&](int t, int kind, uint2 v) {
          const float r = kind == kTokPool ? finish(v.x, __uint_as_float(v.y)) : CUDART_NAN_F;
          if (a.write_stages) rho[t] = r;
          const uint32_t key = kind == kTokPool ? ~float_key(r) : 0u;
          keys[t - j0] = key;
          stats_add(ks, key, 0u);
        });
    // the score phase's inputs arrive in L2 while tau is selected
    if ((a.mode & kSelTopk) && !a.base_uniform) prefetch_l2(a.a_base.at(l) + hn, 4, j0, j1);
    if ((a.mode & kSelTopk) && a.phi.base && a.css_enable) prefetch_l2(a.phi.at(l) + hn, 4, j0, j1);
    if (gate_sel) {
      if (a.tsg_fixed) {
        tau = a.tsg_fixed_tau;  // fixed-threshold control: no selection
        kt_gate = ~float_key(tau);
      } else {
        // the fused call needs only the gated set; the staged call reports tau
        const Selected g = cluster_select(ncta, keys, len, (uint32_t)min(a.budget[l], pool), 0u, ks, sh, 0, pass,
                                          !a.write_stages);
        kt_gate = g.need ? g.T : g.T + 1u;
        tau = key_float(~kt_gate);
      }
    }
    if (c == 0 && tid == 0) a.tau.at(l)[h] = tau;
    __syncthreads();  // the keys are written, also without a select
    if (!(a.mode & kSelTopk)) {
      // gate only: Eq. 8 on the pool, open elsewhere
      for_tokens<2>(
          sh, F, j0, j1, [&](int, int) { return 0; },
          [&](int t, int kind, int) {
            gate[t] = (kind == kTokPool && gate_sel) ? (keys[t - j0] >= kt_gate ? 1 : 0) : 1;
          });
    }
  }

  if (a.mode & kSelTopk) {
    const float* ab = a.base_uniform ? nullptr : a.a_base.at(l) + hn;
    const float* ph = a.phi.base ? a.phi.at(l) + hn : nullptr;
    const uint8_t* gt = gate;
    float* sc = a.score.at(l) + hn;
    const float alpha = a.css_enable ? a.alpha : 0.f;
    const bool fused = (a.mode & kSelGate) != 0;  // gate decided here from the rho keys
    // optional A / max_j A (per head): the cluster-wide maximum first
    float amax = 0.f;
    if (a.a_norm_max) {
      if (ab) {
        float m = 0.f;
        for (int t = j0 + tid; t < j1; t += blockDim.x) m = fmaxf(m, __ldg(ab + t));
        amax = cluster_max(cl, m, sh);
      } else {
        amax = a.a_uniform;
      }
    }
    const bool a_div = amax > 0.f;
    // Eq. 9: S = A_base for text tokens; for visual tokens S = A_base +
    // alpha * Phi where the gate is open and 0 where it is closed
    auto score_of = [&](int t, int kind, float A, float P, float G) {
      float s;
      if (kind == kTokText) {
        s = A + 0.0f;
        if (fused && a.write_stages) gate[t] = 1;
      } else {
        bool g = G != 0.f;
        if (fused) {
          g = !(kind == kTokPool && gate_sel) || keys[t - j0] >= kt_gate;
          if (a.write_stages) gate[t] = g ? 1 : 0;
        }
        const float x = alpha != 0.f ? __fmaf_rn(alpha, P, A) : A;
        s = (g ? x : 0.f) + 0.0f;
      }
      return s;
    };
    const uint32_t zero_key = float_key(0.f);  // a closed gate's score
    stats_init(ks);
    if (vec) {
      for_tokens4(
          sh, F, j0, j1,
          [&](int t0, const int (&kinds)[4]) {
            ScoreIn4 v;
            v.A = ab ? __ldg(reinterpret_cast<const float4*>(ab + t0))
                     : make_float4(a.a_uniform, a.a_uniform, a.a_uniform, a.a_uniform);
            if (a_div)
              v.A = make_float4(__fdiv_rn(v.A.x, amax), __fdiv_rn(v.A.y, amax), __fdiv_rn(v.A.z, amax),
                                __fdiv_rn(v.A.w, amax));
            const bool vis = kinds[0] != kTokText || kinds[1] != kTokText || kinds[2] != kTokText ||
                             kinds[3] != kTokText;
            v.P = (vis && alpha != 0.f) ? __ldg(reinterpret_cast<const float4*>(ph + t0)) : make_float4(0.f, 0.f, 0.f, 0.f);
            v.G = (vis && !fused && gt != nullptr) ? __ldg(reinterpret_cast<const uint32_t*>(gt + t0)) : 0x01010101u;
            return v;
          },
          [&](int t0, const int (&kinds)[4], const ScoreIn4& v) {
            const float s0 = score_of(t0, kinds[0], v.A.x, kinds[0] != kTokText ? v.P.x : 0.f, (float)(v.G & 0xffu));
            const float s1 = score_of(t0 + 1, kinds[1], v.A.y, kinds[1] != kTokText ? v.P.y : 0.f,
                                      (float)((v.G >> 8) & 0xffu));
            const float s2 = score_of(t0 + 2, kinds[2], v.A.z, kinds[2] != kTokText ? v.P.z : 0.f,
                                      (float)((v.G >> 16) & 0xffu));
            const float s3 = score_of(t0 + 3, kinds[3], v.A.w, kinds[3] != kTokText ? v.P.w : 0.f,
                                      (float)(v.G >> 24));
            if (a.write_stages) *reinterpret_cast<float4*>(sc + t0) = make_float4(s0, s1, s2, s3);
            const uint4 kv = make_uint4(float_key(s0), float_key(s1), float_key(s2), float_key(s3));
            *reinterpret_cast<uint4*>(keys + (t0 - j0)) = kv;
            stats_add(ks, kv.x, zero_key);
            stats_add(ks, kv.y, zero_key);
            stats_add(ks, kv.z, zero_key);
            stats_add(ks, kv.w, zero_key);
          });
    } else
    for_tokens<2>(
        sh, F, j0, j1,
        [&](int t, int kind) {
          float A = ab ? __ldg(ab + t) : a.a_uniform;
          if (a_div) A = __fdiv_rn(A, amax);
          const float P = (kind != kTokText && alpha != 0.f) ? __ldg(ph + t) : 0.f;
          const float G = (kind != kTokText && !fused && gt != nullptr) ? (float)gt[t] : 1.f;
          return make_float3(A, P, G);
        },
        [&](int t, int kind, float3 v) {
          const float s = score_of(t, kind, v.x, v.y, v.z);
          if (a.write_stages) sc[t] = s;
          const uint32_t key = float_key(s);
          keys[t - j0] = key;
          stats_add(ks, key, zero_key);
        });
    const Selected top = cluster_select(ncta, keys, len, (uint32_t)a.budget[l], zero_key, ks, sh, 1, pass, true);
    const uint32_t T = top.T, need = top.need;
    // Ordered compaction.  Thread tid owns the contiguous run [r0, r1) of
    // this CTA's keys (odd run length: conflict-free shared reads); one
    // block scan gives its (greater, equal) counts before the run, the
    // cluster's lower ranks add theirs.
    const int per = ((len + (int)blockDim.x - 1) / (int)blockDim.x) | 1;
    const int r0 = min(len, tid * per), r1 = min(len, r0 + per);
    uint32_t g_loc = 0, e_loc = 0;
    for (int i = r0; i < r1; ++i) {
      const uint32_t k = keys[i];
      g_loc += k > T;
      e_loc += k == T;
    }
    uint32_t tot;
    const uint32_t ex = block_exclusive_scan(g_loc | (e_loc << 16), sh.warp_tot, &tot);
    if (tid == 0) {
      sh.counts[0] = tot & 0xffffu;
      sh.counts[1] = tot >> 16;
    }
    cluster_barrier(cl, ncta);
    uint32_t gb = 0, eb = 0;  // of the CTAs before this one
    if ((tid & 31) < c) {
      const uint32_t* rc = cl.map_shared_rank(sh.counts, tid & 31);
      gb = rc[0];
      eb = rc[1];
    }
    uint32_t gt_before = __reduce_add_sync(0xffffffffu, gb) + (ex & 0xffffu);
    uint32_t eq_before = __reduce_add_sync(0xffffffffu, eb) + (ex >> 16);
    int32_t* out = a.idx[l] + (size_t)h * a.budget[l];
    // kept: every key > T, and the first `need` keys == T in index order;
    // a kept token's slot = kept tokens before it
    for (int i = r0; i < r1; ++i) {
      const uint32_t k = keys[i];
      if (k > T) {
        out[gt_before + min(eq_before, need)] = j0 + i;
        ++gt_before;
      } else if (k == T) {
        if (eq_before < need) out[gt_before + eq_before] = j0 + i;
        ++eq_before;
      }
    }
  }
  cluster_barrier(cl, ncta);  // no CTA leaves while a peer may still read its shared memory
}

int select_max_tokens() { return kSelMaxCluster * kSelMaxChunk; }

static int select_chunk(int n, int cl) { return ((n + cl - 1) / cl + 3) & ~3; }

static void select_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr, const Problem& p, int cl,
                          cudaStream_t st) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(cl, p.L * p.hkv, 1);
  cfg->blockDim = dim3(kSelThreads, 1, 1);
  cfg->dynamicSmemBytes = (size_t)select_chunk(p.n, cl) * 4;
  cfg->stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
}

// Clusters of cfg's size and shared memory that are resident at once on device
// dev in the current context (its id; 0: not known): what the occupancy query says of the largest
// shared memory that `occ` CTAs of an SM can have (fit_cache.h), or of cfg
// itself where that says none.
static cudaError_t clusters_fit(int dev, unsigned long long ctx, int c, int occ, int largest,
                                const cudaLaunchConfig_t& cfg, int* fit) {
  static FitCache<64, 2 * kSelMaxCluster, 2048 / kSelThreads> known;
  if ((*fit = known.get(dev, c, occ, ctx)) >= 0) return cudaSuccess;
  cudaLaunchConfig_t ask = cfg;
  ask.dynamicSmemBytes = (size_t)largest;
  cudaError_t e = cudaOccupancyMaxActiveClusters(fit, k_select, &ask);
  if (e == cudaSuccess) known.put(dev, c, occ, ctx, *fit);
  if (e != cudaSuccess || *fit < 1) e = cudaOccupancyMaxActiveClusters(fit, k_select, &cfg);
  return e;
}

cudaError_t launch_select(const Problem& p, const FrameTable& ft, const SelectArgs& a, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_select, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(kSelMaxChunk * 4));
  if (e != cudaSuccess) return e;
  // all of the SM's configurable memory as shared memory: the CTAs' keys
  // are what limits how many clusters are resident
  e = cudaFuncSetAttribute(k_select, cudaFuncAttributePreferredSharedMemoryCarveout,
                           (int)cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  // clusters of 16 (non-portable) where the device takes them
  const bool big = cudaFuncSetAttribute(k_select, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  int nsm = 0, dev = 0, sm_smem = 0, cta_smem = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&cta_smem, cudaDevAttrReservedSharedMemoryPerBlock, dev)) != cudaSuccess) return e;
  cta_smem += (int)sizeof(SelShared);
  unsigned long long ctx = 0;
  if (current_ctx_id(&ctx) != cudaSuccess) ctx = 0;
  // Cluster size: the CTAs of a cluster split one (layer, head)'s tokens.
  // Measured (one wave of clusters, GB300): 13 us for a lone CTA and about
  // 16.5 + 0.55 per CTA for a cluster's barriers and exchanges, plus 1.5 ns per
  // token of a CTA or, where CTAs share SMs, 1.2 ns per token of an SM.  The
  // least sum over the waves wins, the smallest cluster among equals: 28 x 4
  // heads of 53,600 tokens take clusters of 5, which are all resident at once
  // (74 us; 8 need two waves, 98), 28 x 4 of 2,144 single CTAs (20 us; 4: 27),
  // 28 x 2 of 20,000 clusters of 4 (29; 3: 32, 8: 43), 4 of 23,680 clusters of 8
  // (26; 16: 31, 4: 29), 4 of 132,800 clusters of 16 (47; 8: 51).
  // Clusters of 16 only where those of 8 have more than 7,500 tokens a CTA (4
  // heads of 53,600: 35 us, in 16 37; of 90,000: 42 and 39), or more than
  // 28,000 if 16 CTAs would have to share SMs, which they do from the eighth
  // cluster on (8 heads of 53,600: 35 us, in 16 43; of 132,800: 51 and 55; of
  // 260,000: 78 and 76).
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  int cl = 0;
  double best = 0.0;
  const long long units = (long long)p.L * p.hkv;
  for (int c = 1; c <= (big ? 2 : 1) * kSelMaxCluster; c = c < kSelMaxCluster ? c + 1 : 2 * c) {
    const int ch = select_chunk(p.n, c);
    if (ch > kSelMaxChunk) continue;
    select_config(&cfg, attr, p, c, st);
    const int occ = ctas_per_sm(sm_smem, cta_smem, 4 * ch, 2048 / kSelThreads);
    if (occ < 1) continue;
    int fit = 0;
    const int largest = largest_dynamic(sm_smem, cta_smem, occ, 4 * kSelMaxChunk);
    if ((e = clusters_fit(dev, ctx, c, occ, largest, cfg, &fit)) != cudaSuccess) {
      if (c <= kSelMaxCluster) return e;
      break;
    }
    if (fit < 1) continue;
    if (c > kSelMaxCluster && cl != 0) {
      int alone = 0;  // clusters whose CTAs have an SM each
      const int own = largest_dynamic(sm_smem, cta_smem, 1, 4 * kSelMaxChunk);
      if ((e = clusters_fit(dev, ctx, c, 1, own, cfg, &alone)) != cudaSuccess) break;
      if (select_chunk(p.n, kSelMaxCluster) <= (units <= alone ? 7500 : 28000)) break;
    }
    const double fixed = c == 1 ? 13.0 : 16.5 + 0.55 * c;
    double cost = 0.0;
    for (long long left = units; left > 0; left -= fit) {
      const double per_sm = (double)std::min<long long>(left, fit) * c * ch / nsm;
      cost += fixed + std::max(1.5e-3 * ch, 1.2e-3 * per_sm);
    }
    if (cl == 0 || cost < best) {
      cl = c;
      best = cost;
    }
  }
  (void)cudaGetLastError();  // a refused non-portable query leaves no error behind
  if (cl == 0) return cudaErrorNotSupported;
  select_config(&cfg, attr, p, cl, st);
  TimingScope ts(a.mode & kSelGate ? (a.mode & kSelTopk ? "select_gate_topk" : "select_gate") : "select_topk", st);
  e = cudaLaunchKernelEx(&cfg, k_select, p, ft, a);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

// ------------------------------------------------------------------ gather
// k_out[l][r][h][:] = k_l[idx[l][h][r]][h][:] (and v): 16-byte chunks, four
// rows per thread in flight, consecutive threads cover consecutive chunks of
// one output row (coalesced stores, whole 16-byte source vectors).  Plain
// loads: idx, and whatever else the kernel before it wrote, was written while
// this one was already resident (and v may be page-locked host memory).
// grid.y = layer.
template <int CPR>
__global__ void __launch_bounds__(256) k_gather(const __grid_constant__ LayerPtrs io, int n, int hkv) {
  pdl_wait();
  const int l = blockIdx.y;
  const int budget = io.budget[l];
  const int32_t* idx = io.idx[l];
  const uint4* k = static_cast<const uint4*>(io.k[l]);
  const uint4* v = static_cast<const uint4*>(io.v[l]);
  uint4* ko = static_cast<uint4*>(io.k_out[l]);
  uint4* vo = static_cast<uint4*>(io.v_out[l]);
  const long long total = (long long)budget * hkv * CPR;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long e0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; e0 < total; e0 += 4 * stride) {
    uint4 kv[4], vv[4];
    long long ee[4];
    bool ok[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long long e = e0 + u * stride;
      ee[u] = e;
      ok[u] = false;
      if (e < total) {
        const int c = (int)(e % CPR);
        const long long rh = e / CPR;
        const int h = (int)(rh % hkv), r = (int)(rh / hkv);
        const int src = idx[(size_t)h * budget + r];
        if (src >= 0 && src < n) {
          const size_t s = ((size_t)src * hkv + h) * CPR + c;
          kv[u] = k[s];
          vv[u] = v[s];
          ok[u] = true;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (ok[u]) {
        ko[ee[u]] = kv[u];
        vo[ee[u]] = vv[u];
      }
    }
  }
}

cudaError_t launch_gather(const Problem& p, const LayerPtrs& io, cudaStream_t st) {
  const int cpr = p.dtype == kBF16 ? kD * 2 / 16 : kD * 4 / 16;
  int bmax = 1;
  for (int l = 0; l < p.L; ++l) bmax = io.budget[l] > bmax ? io.budget[l] : bmax;
  long long total = (long long)bmax * p.hkv * cpr;
  long long blocks = (total + 1023) / 1024;
  long long cap = (152 * 8 + p.L - 1) / p.L;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  TimingScope ts("gather", st);
  dim3 grid((unsigned)blocks, p.L);
  const cudaError_t e = launch_after(cpr == 16 ? k_gather<16> : k_gather<32>, grid, 256, 0, st, io, p.n, p.hkv);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace stl
