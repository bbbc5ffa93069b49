// Products of two sets of 128-wide fp32 rows on the CUDA cores, and the
// online softmax over their results: the parts shared by the fp32 passes.
#pragma once

#include "common.cuh"

namespace stl {

// ------------------------------------------------ fp32 tile products
// The fp32 passes below are products of two sets of 128-wide rows, bound by
// the FMA pipe.  A CTA of 128 threads forms the 64 x 64 dot products of two
// row sets in shared memory (rows padded to 132 floats, so that a warp's four
// rows of A or eight of B lie in different banks), eight x four per thread:
// per four dimensions, twelve 16-byte shared loads feed 64 packed
// multiply-adds.  67.6 KB let three CTAs share an SM; one's copies hide behind
// the others' products.  Even and odd dimensions accumulate apart (the two
// halves of fma.rn.f32x2), each in ascending order, and are added last.
// The product alone reaches 50 TFLOP/s of the FMA pipe's 76 (8 x 8 per thread:
// 52, but two CTAs of half the warps; 4 x 8: 48; unpacked fmaf: the same).
// One layer of 5 frames of 36 x 64 (11,840 keys, 4 heads of 224 query rows),
// against one dot product per thread with both operands read from shared
// memory for every multiply-add: TSG 2,036 -> 483 us (45 TFLOP/s), row
// statistics 389 -> 94, column sums 466 -> 92; 1,152 keys: 201 -> 15, 90 -> 18
// and 195 -> 29 (17 with a cluster per key tile, simt.cu).
constexpr int kTileRows = 64;
constexpr int kTileThreads = 128;
constexpr int kTilePitch = kD + 4;  // floats
constexpr int kTileFloats = kTileRows * kTilePitch;
constexpr int kTA = 8, kTB = 4;  // rows of A and B per thread
constexpr int kTilesPerSm = 3;

// The thread's rows: ty + 8 i of A, tx + 16 j of B.  A warp holds four ty
// and eight tx; warps 2 and 3 have the other four ty, odd warps the other tx.
__device__ __forceinline__ int tile_ty() { return ((threadIdx.x >> 3) & 3) + 4 * (threadIdx.x >> 6); }
__device__ __forceinline__ int tile_tx() { return (threadIdx.x & 7) + 8 * ((threadIdx.x >> 5) & 1); }

// Starts the copy of rows src(0) .. src(nrows - 1) (512 bytes each) into a
// tile; the rows after them become zero.  A warp copies one row at a time.
template <class Src>
__device__ __forceinline__ void tile_load(float* dst, int nrows, Src src) {
  const int lane = threadIdx.x & 31;
#pragma unroll 4
  for (int r = threadIdx.x >> 5; r < kTileRows; r += kTileThreads / 32) {
    float* d = dst + r * kTilePitch + 4 * lane;
    if (r < nrows) {
      const uint32_t da = static_cast<uint32_t>(__cvta_generic_to_shared(d));
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(da), "l"(src(r) + 4 * lane) : "memory");
    } else {
      *reinterpret_cast<float4*>(d) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
}
// Every copy of the CTA has landed (and every thread's use of the tiles
// before this call is over).
__device__ __forceinline__ void tile_ready() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
  __syncthreads();
}

// d[i][j] = A row (ty + 8 i) . B row (tx + 16 j)
__device__ __forceinline__ void tile_dots(const float* a, const float* b, float (&d)[kTA][kTB]) {
  const float* ap = a + tile_ty() * kTilePitch;
  const float* bp = b + tile_tx() * kTilePitch;
  unsigned long long acc[kTA][kTB];
#pragma unroll
  for (int i = 0; i < kTA; ++i)
#pragma unroll
    for (int j = 0; j < kTB; ++j) acc[i][j] = 0ull;
#pragma unroll 4
  for (int k = 0; k < kD; k += 4) {
    ulonglong2 y[kTB];
#pragma unroll
    for (int j = 0; j < kTB; ++j) y[j] = *reinterpret_cast<const ulonglong2*>(bp + 16 * j * kTilePitch + k);
#pragma unroll
    for (int i = 0; i < kTA; ++i) {
      const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(ap + 8 * i * kTilePitch + k);
#pragma unroll
      for (int j = 0; j < kTB; ++j) {
        asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[i][j]) : "l"(x.x), "l"(y[j].x));
        asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[i][j]) : "l"(x.y), "l"(y[j].y));
      }
    }
  }
#pragma unroll
  for (int i = 0; i < kTA; ++i)
#pragma unroll
    for (int j = 0; j < kTB; ++j) {
      float lo, hi;
      asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(acc[i][j]));
      d[i][j] = lo + hi;
    }
}

// s.x + s.y += x, the rounding error of the sum s.x kept in s.y (Knuth's
// two-sum).
__device__ __forceinline__ void add_exact(float2& s, float x) {
  const float t = s.x + x, b = t - s.x;
  s.y += (s.x - (t - b)) + (x - b);
  s.x = t;
}
__device__ __forceinline__ void add_exact(float2& s, float2 x) {
  add_exact(s, x.x);
  s.y += x.y;
}

// (m, l) <- the states (m, l) and (m2, l2) together; l = 0: an empty state.
__device__ __forceinline__ void merge_state(float& m, float& l, float m2, float l2) {
  if (l2 == 0.f) return;
  if (l == 0.f) {
    m = m2;
    l = l2;
    return;
  }
  const float mn = fmaxf(m, m2);
  l = (m == mn ? l : l * exp2f(m - mn)) + (m2 == mn ? l2 : l2 * exp2f(m2 - mn));
  m = mn;
}

// (m, l) <- (m, l) and the scores x[0..kTB-1] (log2 units; -inf: none).  m is
// the maximum rounded up to a whole number, so that every later change of m,
// here or when states merge, scales l by a power of two, without rounding.
// With the maximum itself, and plain sums of the probabilities, the scores of
// few rows were up to 26 % further from the fp64 result than one thread's sums
// over a row had been; with this and add_exact they are 1.4-8 times nearer (one
// row per head: the same), at 3 % of the column sums' time.
__device__ __forceinline__ void fold_scores(float& m, float& l, const float (&x)[kTB]) {
  float mn = m;
#pragma unroll
  for (int j = 0; j < kTB; ++j) mn = fmaxf(mn, x[j]);
  if (mn == -CUDART_INF_F) return;  // no score yet
  mn = ceilf(mn);
  float sum = 0.f;
#pragma unroll
  for (int j = 0; j < kTB; ++j) sum += x[j] == mn ? 1.f : exp2f(x[j] - mn);
  l = (m == mn ? l : l * exp2f(m - mn)) + sum;
  m = mn;
}

// The states of the CTA's rows, merged over the sixteen threads that share a
// row: eight lanes of each of two warps.  The threads with tile_tx() == 0 end
// with row ty + 8 i's state in m[i], l[i].  xch: a tile's worth of shared
// memory that nobody reads any more once every thread has come here.
__device__ __forceinline__ void merge_rows(float (&m)[kTA], float (&l)[kTA], float* xch) {
  const int ty = tile_ty(), tx = tile_tx();
#pragma unroll
  for (int i = 0; i < kTA; ++i)
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m[i], o), l2 = __shfl_xor_sync(0xffffffffu, l[i], o);
      merge_state(m[i], l[i], m2, l2);
    }
  tile_ready();  // also without a tile: copies still in flight end before the CTA does
  float2* x = reinterpret_cast<float2*>(xch);
  if (tx == 8)
#pragma unroll
    for (int i = 0; i < kTA; ++i) x[ty + 8 * i] = make_float2(m[i], l[i]);
  __syncthreads();
  if (tx == 0)
#pragma unroll
    for (int i = 0; i < kTA; ++i) {
      const float2 o = x[ty + 8 * i];
      merge_state(m[i], l[i], o.x, o.y);
    }
}

// Sums per row with their rounding errors (add_exact), merged the same way, into
// sums[0..63] (shared memory, as xch above); a block barrier away from being read.
__device__ __forceinline__ void sum_rows(float2 (&acc)[kTA], float2* sums) {
  const int ty = tile_ty(), tx = tile_tx();
#pragma unroll
  for (int i = 0; i < kTA; ++i)
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      const float x = __shfl_xor_sync(0xffffffffu, acc[i].x, o), y = __shfl_xor_sync(0xffffffffu, acc[i].y, o);
      add_exact(acc[i], make_float2(x, y));
    }
  tile_ready();
  if (tx == 8)
#pragma unroll
    for (int i = 0; i < kTA; ++i) sums[ty + 8 * i] = acc[i];
  __syncthreads();
  if (tx == 0)
#pragma unroll
    for (int i = 0; i < kTA; ++i) {
      add_exact(acc[i], sums[ty + 8 * i]);
      sums[ty + 8 * i] = acc[i];
    }
}

}  // namespace stl
