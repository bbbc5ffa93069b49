// Device-side helpers shared by every ST-Lite kernel (sm_103a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

namespace stl {

constexpr int kD = 128;            // head dimension handled by every kernel
constexpr int kMaxFrames = 256;    // frames per sequence
constexpr int kTsgTile = 128;      // historical tokens per TSG row tile

// Device error word bits (first 32-bit word of the workspace).
constexpr uint32_t kErrTimeout = 1u;  // a bounded wait ran out
constexpr uint32_t kErrLaunch = 2u;   // a kernel found its launch configuration unusable

// Bounded waits give up after this many nanoseconds of %globaltimer.
constexpr uint64_t kWaitLimitNs = 1000000000ull;

// Frame layout of one sequence, passed by value (__grid_constant__) so that
// no host-to-device copy is needed.  Frame f owns tokens
// [off[f], off[f] + gh[f]*gw[f]); the last frame is the current frame.
// tile0[f] is the index of the first 128-token TSG row tile of historical
// frame f (tile0[F-1] = total tiles over frames 0..F-2).
struct FrameTable {
  int32_t n_frames;
  int32_t n_tokens;
  int32_t cur_off;   // first token of the current frame (0 if F == 0)
  int32_t cur_len;   // its visual token count (0 if F == 0)
  int32_t off[kMaxFrames];
  int32_t gh[kMaxFrames];
  int32_t gw[kMaxFrames];
  int32_t tile0[kMaxFrames + 1];
  int32_t ctile0[kMaxFrames + 1];  // first 128-token CSS tile of every frame (all frames)
  // Row tiles of the tensor-core TSG pass: per historical frame (tile0), or,
  // when that takes more tiles, 128-token tiles spanning the whole range
  // [tsg_off, tsg_end) of the historical frames, text tokens included (their
  // rho slices are never read).
  int32_t tsg_tiles;
  int32_t tsg_span;  // 1: spanning tiles
  int32_t tsg_off, tsg_end;
};

// Frame holding token j, or -1 for a text token (binary search on offsets).
__device__ __forceinline__ int find_frame(const FrameTable& ft, int j) {
  int lo = 0, hi = ft.n_frames - 1, f = -1;
  while (lo <= hi) {
    int mid = (lo + hi) >> 1;
    if (ft.off[mid] <= j) {
      f = mid;
      lo = mid + 1;
    } else {
      hi = mid - 1;
    }
  }
  if (f >= 0 && j < ft.off[f] + ft.gh[f] * ft.gw[f]) return f;
  return -1;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Folds one split partial (m2, l2) of the window score's row statistics into
// (m, l): the running max in log2 units and the sum of 2^(x - max).
// Symmetric in its two arguments, bit for bit (max and a two-term sum commute).
__device__ __forceinline__ void fold_partial(float& m, float& l, float m2, float l2) {
  if (!(l2 > 0.f)) return;
  if (!(l > 0.f)) {
    m = m2;
    l = l2;
    return;
  }
  const float mn = fmaxf(m, m2);
  l = l * exp2f(m - mn) + l2 * exp2f(m2 - mn);
  m = mn;
}

// The bias -m - log2(G l) of one query row from its splits' partials pp[0],
// pp[R], pp[2 R], ..., by four neighbouring lanes (whole warps call it): lane q
// folds splits q, q + 4, q + 8, ... (eight loads in flight), then the four
// lanes' states are folded pairwise with shuffles, so that every lane holds
// the same bits.  The order depends on the split count alone.
__device__ __forceinline__ float row_bias4(const float2* pp, int R, int nsplit, float G) {
  const int q = threadIdx.x & 3;
  float m = -CUDART_INF_F, l = 0.f;
  for (int s0 = q; s0 < nsplit; s0 += 32) {
    float2 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      v[u] = s0 + 4 * u < nsplit ? pp[(size_t)(s0 + 4 * u) * R] : make_float2(-CUDART_INF_F, 0.f);
#pragma unroll
    for (int u = 0; u < 8; ++u) fold_partial(m, l, v[u].x, v[u].y);
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, o), l2 = __shfl_xor_sync(0xffffffffu, l, o);
    fold_partial(m, l, m2, l2);
  }
  return -m - log2f(G * l);
}

// Order-preserving map float -> uint32 (ascending keys = ascending floats).
// -0.0 is folded onto +0.0 first so that the two compare equal, as they do
// as numbers.
__device__ __forceinline__ uint32_t float_key(float x) {
  uint32_t u = __float_as_uint(x + 0.0f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k) {
  uint32_t u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
  return __uint_as_float(u);
}

__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Programmatic dependent launch (launch_after): a kernel launched that way may
// start while its predecessor in the stream still runs; pdl_wait returns once
// the predecessor has completed and its writes are visible, and pdl_trigger
// lets a successor start.  Every thread of such a kernel waits, so it completes
// after its predecessor does and the order of the stream holds for whatever
// follows.  Before the wait it touches no global memory, with one exception:
// k_colsum_umma, which reads q and k (see launch_score_umma).  And since it is
// resident while its predecessor still writes, it reads with plain or
// asynchronous loads only, never through the read-only path.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void record_error(uint32_t* err, uint32_t bits) {
  if (err) atomicOr(err, bits);
}

}  // namespace stl
