// CUDA-core kernels: inverse key norms, CSS saliency, and the fp32 versions
// of window scoring and TSG (fp32 inputs cannot use the bf16 tensor-core
// path without losing the exactness of the products).  Every kernel covers a
// batch of layers: the layer index is the high part of one grid dimension.
#include <cooperative_groups.h>

#include "kernels.cuh"
#include "tile.cuh"

namespace cg = cooperative_groups;

namespace stl {

constexpr float kLog2e = 1.4426950408889634f;

// 16 bytes of keys -> floats (8 bf16 or 4 fp32).  Shared by the norm and CSS
// kernels, so that both compute a key's norm with the same sequence of
// operations (fmaf over elements 0..127 in order) and agree bit for bit.
template <typename T>
__device__ __forceinline__ void unpack16(const uint4& w, float (&f)[16 / sizeof(T)]) {
  if constexpr (sizeof(T) == 2) {
    f[0] = __uint_as_float(w.x << 16);
    f[1] = __uint_as_float(w.x & 0xffff0000u);
    f[2] = __uint_as_float(w.y << 16);
    f[3] = __uint_as_float(w.y & 0xffff0000u);
    f[4] = __uint_as_float(w.z << 16);
    f[5] = __uint_as_float(w.z & 0xffff0000u);
    f[6] = __uint_as_float(w.w << 16);
    f[7] = __uint_as_float(w.w & 0xffff0000u);
  } else {
    f[0] = __uint_as_float(w.x);
    f[1] = __uint_as_float(w.y);
    f[2] = __uint_as_float(w.z);
    f[3] = __uint_as_float(w.w);
  }
}

// ---------------------------------------------------------------- norms
// rn[l][h][j] = 1 / max(|k_l[j,h]|, 1e-8); one thread per (token, head) row,
// grid.y = layer.
template <typename T>
__global__ void __launch_bounds__(256) k_inv_norms(const __grid_constant__ LayerPtrs io, int n, int hkv,
                                                   NormsOut norms, int cur_off, int cur_len) {
  constexpr int kChunks = kD * (int)sizeof(T) / 16;
  constexpr int kPer = 16 / (int)sizeof(T);
  const int l = blockIdx.y;
  const T* k = static_cast<const T*>(io.k[l]);
  float* rn = norms.rn.at(l);
  uint32_t* rho = norms.rho_key.base ? norms.rho_key.at(l) : nullptr;
  const long long rows = (long long)n * hkv;
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < rows;
       r += (long long)gridDim.x * blockDim.x) {
    const uint4* src = reinterpret_cast<const uint4*>(k + r * kD);
    uint4 w[kChunks];
#pragma unroll
    for (int c = 0; c < kChunks; ++c) w[c] = __ldg(src + c);
    float sn = 0.f;
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
      float x[kPer];
      unpack16<T>(w[c], x);
#pragma unroll
      for (int t = 0; t < kPer; ++t) sn = fmaf(x[t], x[t], sn);
    }
    const long long j = r / hkv, h = r - j * hkv;
    const float v = 1.0f / fmaxf(sqrtf(sn), 1e-8f);
    rn[h * n + j] = v;
    if (rho) rho[h * n + j] = 0u;
    if (j >= cur_off && j < cur_off + cur_len) norms.rn_cur.at(l)[h * norms.cur_pad + (j - cur_off)] = v;
  }
}

cudaError_t launch_inv_norms(const Problem& p, const FrameTable& ft, const LayerPtrs& io, const NormsOut& norms,
                             cudaStream_t st) {
  long long rows = (long long)p.n * p.hkv;
  long long blocks = (rows + 255) / 256;
  long long cap = (152 * 8 + p.L - 1) / p.L;
  if (blocks > cap) blocks = cap;
  TimingScope ts("inv_norms", st);
  dim3 grid((unsigned)blocks, p.L);
  if (p.dtype == kBF16)
    k_inv_norms<__nv_bfloat16><<<grid, 256, 0, st>>>(io, p.n, p.hkv, norms, ft.cur_off, ft.cur_len);
  else
    k_inv_norms<float><<<grid, 256, 0, st>>>(io, p.n, p.hkv, norms, ft.cur_off, ft.cur_len);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- CSS
// Eqs. 4-5 on 2-D tiles of one frame's patch grid.  A CTA (tile, frame,
// layer*Hkv + head) stages the tile's keys plus a one-cell halo in shared
// memory with asynchronous copies (key rows padded by 16 bytes, so 8 threads
// reading 8 different keys hit 8 distinct bank groups).  One thread per cell
// then computes the cell's norm and its E, S, SE, SW pair dots in one sweep,
// so every unordered neighbour pair is computed once; finally each output
// cell sums its eight directions.  The inverse norms of the output cells are
// written too (TSG uses them).
constexpr int kCssThreads = 256;
constexpr int kCssBudget = 100 * 1024;  // shared-memory bytes per CTA
constexpr int kCssMaxCols = 64;         // output columns per tile

template <typename T>
struct CssGeom {
  static constexpr int kStride = kD * (int)sizeof(T) + 16;   // padded key row
  static constexpr int kCellBytes = kStride + 5 * 4;         // key + rn + 4 pair dots
  static constexpr int kCap = kCssBudget / kCellBytes;       // cells per CTA
  // output tile of CB columns x RB rows, loaded as (RB+2) x (CB+2) cells
  __host__ __device__ static void tile(int gh, int gw, int& RB, int& CB) {
    CB = gw < kCssMaxCols ? gw : kCssMaxCols;
    RB = kCap / (CB + 2) - 2;
    if (RB < 1) RB = 1;
    if (RB > gh) RB = gh;
  }
  __host__ __device__ static int tiles(int gh, int gw) {
    int RB, CB;
    tile(gh, gw, RB, CB);
    return ((gh + RB - 1) / RB) * ((gw + CB - 1) / CB);
  }
};

template <typename T>
__global__ void __launch_bounds__(kCssThreads) k_css(const __grid_constant__ LayerPtrs io,
                                                     const __grid_constant__ FrameTable ft, int hkv,
                                                     Strided<float> phi_all, NormsOut norms) {
  using Gm = CssGeom<T>;
  constexpr int kChunks = kD * (int)sizeof(T) / 16;
  constexpr int kPer = 16 / (int)sizeof(T);
  extern __shared__ float4 css_smem[];
  uint8_t* sm = reinterpret_cast<uint8_t*>(css_smem);
  const int f = blockIdx.y, l = blockIdx.z / hkv, h = blockIdx.z % hkv, n = ft.n_tokens;
  const int tid = threadIdx.x;
  if (f >= ft.n_frames) return;
  const T* k = static_cast<const T*>(io.k[l]);
  float* phi = phi_all.at(l);
  float* rn_out = norms.rn.at(l);
  const int gh = ft.gh[f], gw = ft.gw[f], off = ft.off[f];
  int RB, CB;
  Gm::tile(gh, gw, RB, CB);
  const int tv = (gw + CB - 1) / CB;
  if ((int)blockIdx.x >= ((gh + RB - 1) / RB) * tv) return;
  const int u0 = ((int)blockIdx.x / tv) * RB, v0 = ((int)blockIdx.x % tv) * CB;
  const int TW = CB + 2, TH = RB + 2, cells = TW * TH;
  uint8_t* keys = sm;
  float* rn = reinterpret_cast<float*>(sm + (size_t)cells * Gm::kStride);
  float* dE = rn + cells;
  float* dS = dE + cells;
  float* dSE = dS + cells;
  float* dSW = dSE + cells;
  // stage the tile (local cell (a, b) = grid cell (u0 - 1 + a, v0 - 1 + b));
  // cells outside the grid stay unloaded and are never read
  for (int e = tid; e < cells * kChunks; e += blockDim.x) {
    const int cell = e / kChunks, ch = e - cell * kChunks;
    const int u = u0 - 1 + cell / TW, v = v0 - 1 + cell % TW;
    if (u < 0 || u >= gh || v < 0 || v >= gw) continue;
    const T* src = k + ((size_t)(off + u * gw + v) * hkv + h) * kD + ch * kPer;
    const uint32_t dst =
        static_cast<uint32_t>(__cvta_generic_to_shared(keys + (size_t)cell * Gm::kStride + 16 * ch));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  }
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // one thread per cell: its norm and its E, S, SE, SW pair dots in one sweep
  // (a missing partner reads the cell itself and is discarded)
  for (int cell = tid; cell < cells; cell += blockDim.x) {
    const int a = cell / TW, b = cell % TW;
    const int u = u0 - 1 + a, v = v0 - 1 + b;
    if (u < 0 || u >= gh || v < 0 || v >= gw) continue;
    const bool fwd = a <= RB && u + 1 < gh;
    const bool hasE = b + 1 < TW && v + 1 < gw;
    const bool hasSE = fwd && b + 1 < TW && v + 1 < gw;
    const bool hasSW = fwd && b >= 1 && v >= 1;
    const uint8_t* p0 = keys + (size_t)cell * Gm::kStride;
    const uint8_t* pE = hasE ? p0 + Gm::kStride : p0;
    const uint8_t* pS = fwd ? p0 + (size_t)TW * Gm::kStride : p0;
    const uint8_t* pSE = hasSE ? p0 + (size_t)(TW + 1) * Gm::kStride : p0;
    const uint8_t* pSW = hasSW ? p0 + (size_t)(TW - 1) * Gm::kStride : p0;
    float sn = 0.f, sE = 0.f, sS = 0.f, sSE = 0.f, sSW = 0.f;
#pragma unroll 4
    for (int c = 0; c < kChunks; ++c) {
      float x[kPer], y[kPer];
      unpack16<T>(*reinterpret_cast<const uint4*>(p0 + 16 * c), x);
#pragma unroll
      for (int t = 0; t < kPer; ++t) sn = fmaf(x[t], x[t], sn);
      unpack16<T>(*reinterpret_cast<const uint4*>(pE + 16 * c), y);
#pragma unroll
      for (int t = 0; t < kPer; ++t) sE = fmaf(x[t], y[t], sE);
      unpack16<T>(*reinterpret_cast<const uint4*>(pS + 16 * c), y);
#pragma unroll
      for (int t = 0; t < kPer; ++t) sS = fmaf(x[t], y[t], sS);
      unpack16<T>(*reinterpret_cast<const uint4*>(pSE + 16 * c), y);
#pragma unroll
      for (int t = 0; t < kPer; ++t) sSE = fmaf(x[t], y[t], sSE);
      unpack16<T>(*reinterpret_cast<const uint4*>(pSW + 16 * c), y);
#pragma unroll
      for (int t = 0; t < kPer; ++t) sSW = fmaf(x[t], y[t], sSW);
    }
    rn[cell] = 1.0f / fmaxf(sqrtf(sn), 1e-8f);
    dE[cell] = sE;
    dS[cell] = sS;
    dSE[cell] = sSE;
    dSW[cell] = sSW;
  }
  __syncthreads();
  for (int o = tid; o < RB * CB; o += blockDim.x) {
    const int u = u0 + o / CB, v = v0 + o % CB;
    if (u >= gh || v >= gw) continue;
    const int c = (o / CB + 1) * TW + (o % CB + 1);
    const float r0 = rn[c];
    float sum = 0.f;
    int cnt = 0;
    const bool up = u > 0, dn = u + 1 < gh, lf = v > 0, rt = v + 1 < gw;
    if (rt) { sum += dE[c] * r0 * rn[c + 1]; ++cnt; }
    if (lf) { sum += dE[c - 1] * rn[c - 1] * r0; ++cnt; }
    if (dn) { sum += dS[c] * r0 * rn[c + TW]; ++cnt; }
    if (up) { sum += dS[c - TW] * rn[c - TW] * r0; ++cnt; }
    if (dn && rt) { sum += dSE[c] * r0 * rn[c + TW + 1]; ++cnt; }
    if (up && lf) { sum += dSE[c - TW - 1] * rn[c - TW - 1] * r0; ++cnt; }
    if (dn && lf) { sum += dSW[c] * r0 * rn[c + TW - 1]; ++cnt; }
    if (up && rt) { sum += dSW[c - TW + 1] * rn[c - TW + 1] * r0; ++cnt; }
    const int j = off + u * gw + v;
    phi[(size_t)h * n + j] = cnt ? 1.0f - sum / (float)cnt : 0.0f;
    rn_out[(size_t)h * n + j] = r0;
    if (norms.rho_key.base) norms.rho_key.at(l)[(size_t)h * n + j] = 0u;
    if (f == ft.n_frames - 1) norms.rn_cur.at(l)[(size_t)h * norms.cur_pad + (j - off)] = r0;
  }
}

// Phi of text tokens is undefined: NaN (only the staged entry point writes it).
__global__ void k_fill_text_nan(const __grid_constant__ FrameTable ft, int hkv, float* __restrict__ phi) {
  const int n = ft.n_tokens;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < (long long)n * hkv;
       e += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(e % n);
    if (find_frame(ft, j) < 0) phi[e] = CUDART_NAN_F;
  }
}

template <typename T>
static cudaError_t css_launch_t(const Problem& p, const FrameTable& ft, const LayerPtrs& io,
                                Strided<float> phi, const NormsOut& norms, cudaStream_t st) {
  using Gm = CssGeom<T>;
  int tmax = 0, cmax = 0;
  for (int f = 0; f < ft.n_frames; ++f) {
    int RB, CB;
    Gm::tile(ft.gh[f], ft.gw[f], RB, CB);
    tmax = max(tmax, Gm::tiles(ft.gh[f], ft.gw[f]));
    cmax = max(cmax, (RB + 2) * (CB + 2));
  }
  if (tmax == 0) return cudaSuccess;
  const size_t smem = (size_t)cmax * Gm::kCellBytes;
  cudaError_t e = cudaFuncSetAttribute(k_css<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  TimingScope ts("css", st);
  k_css<T><<<dim3(tmax, ft.n_frames, p.L * p.hkv), kCssThreads, smem, st>>>(io, ft, p.hkv, phi, norms);
  return cudaGetLastError();
}

cudaError_t launch_css(const Problem& p, const FrameTable& ft, const LayerPtrs& io, Strided<float> phi,
                       const NormsOut& norms, cudaStream_t st) {
  if (p.dtype == kBF16) return css_launch_t<__nv_bfloat16>(p, ft, io, phi, norms, st);
  return css_launch_t<float>(p, ft, io, phi, norms, st);
}

// ------------------------------------------------------- CSS, k x k box
// Eqs. 4-5 over the (2R+1) x (2R+1) neighbourhood (R = 1 is the method's 3x3
// Moore neighbourhood; R = 2..4 the 5x5..9x9 kernels of the size ablation).
// With khat_j = k_j / max(|k_j|, 1e-8) the neighbour cosines add up to
//   sum_{j in N(i)} cos(k_i, k_j) = khat_i . (sum_{j in box(i)} khat_j - khat_i),
// so a cell needs one box sum of normalised keys, whatever the size, and
// the box sum separates into row sums and a sum of 2R+1 rows.  A CTA (tile,
// frame, layer*Hkv + head) stages kBoxRows x kBoxCols output cells plus an
// R-cell halo (out-of-grid cells as zero keys with rn = 0, so they add
// nothing); 16 or 32 lanes own a pair of adjacent output columns, walk the
// tile's rows once and keep the last 2R+1 row sums in registers.  rn of a cell
// uses the same operation sequence as the norms kernel, so both agree bit for
// bit.  Bound by issue slots and shared-memory reads: a pair reads a row's
// 2R+2 cells once where two single columns read 4R+2, and the sums use packed
// fp32x2 operations (each half rounded as a scalar one).  5x5 over 28 layers
// of 53,600 bf16 tokens: 1,141 -> 925 us; 9x9: 2,000 -> 1,640; fp32, 23,104
// tokens: 61 -> 52 us.  16 lanes (8 dimensions each) for the small bf16 boxes;
// else 32: with twice the warps and half the registers 7x7 takes 1,320 us, not
// 1,426, and fp32, whose 127 KB tile leaves one CTA per SM, 52 us, not 71 (5x5
// bf16: 987, not 925).
constexpr int kBoxRows = 8, kBoxCols = 16;

// two fp32 values of a packed fp32x2 operand, first in the low half
__device__ __forceinline__ uint64_t pack_f2(float x, float y) {
  return (uint64_t)__float_as_uint(y) << 32 | __float_as_uint(x);
}
__device__ __forceinline__ float2 unpack_f2(uint64_t v) {
  return make_float2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)));
}

template <typename T, int R>
struct BoxGeom {
  static constexpr int TH = kBoxRows + 2 * R, TW = kBoxCols + 2 * R, cells = TH * TW;
  static constexpr int stride = kD * (int)sizeof(T) + 16;  // padded key row
  static constexpr int smem = cells * stride + cells * 4;
  static constexpr int lanes = sizeof(T) == 2 && R <= 2 ? 16 : 32;  // of a pair of columns
  static constexpr int threads = kBoxCols / 2 * lanes;
};

template <typename T, int R>
__global__ void __launch_bounds__(BoxGeom<T, R>::threads) k_css_box(const __grid_constant__ LayerPtrs io,
                                                         const __grid_constant__ FrameTable ft, int hkv,
                                                         Strided<float> phi_all, NormsOut norms) {
  using Gm = BoxGeom<T, R>;
  constexpr int kChunks = kD * (int)sizeof(T) / 16;
  constexpr int kPer = 16 / (int)sizeof(T);
  constexpr int TW = Gm::TW, TH = Gm::TH, D2 = 2 * R + 1, kLanes = Gm::lanes;
  extern __shared__ float4 box_smem[];
  uint8_t* keys = reinterpret_cast<uint8_t*>(box_smem);
  float* rn = reinterpret_cast<float*>(keys + (size_t)Gm::cells * Gm::stride);
  const int f = blockIdx.y, l = blockIdx.z / hkv, h = blockIdx.z % hkv, n = ft.n_tokens;
  const int tid = threadIdx.x;
  if (f >= ft.n_frames) return;
  const int gh = ft.gh[f], gw = ft.gw[f], off = ft.off[f];
  const int tv = (gw + kBoxCols - 1) / kBoxCols;
  if ((int)blockIdx.x >= ((gh + kBoxRows - 1) / kBoxRows) * tv) return;
  const int u0 = ((int)blockIdx.x / tv) * kBoxRows, v0 = ((int)blockIdx.x % tv) * kBoxCols;
  const T* k = static_cast<const T*>(io.k[l]);
  // stage: local cell (a, b) = grid cell (u0 - R + a, v0 - R + b)
  for (int e = tid; e < Gm::cells * kChunks; e += blockDim.x) {
    const int cell = e / kChunks, ch = e - cell * kChunks;
    const int u = u0 - R + cell / TW, v = v0 - R + cell % TW;
    uint8_t* dstp = keys + (size_t)cell * Gm::stride + 16 * ch;
    if (u < 0 || u >= gh || v < 0 || v >= gw) {
      *reinterpret_cast<uint4*>(dstp) = make_uint4(0u, 0u, 0u, 0u);
      continue;
    }
    const T* src = k + ((size_t)(off + u * gw + v) * hkv + h) * kD + ch * kPer;
    const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(dstp));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  }
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // inverse norms (0 outside the grid); the output cells' go to rn / rn_cur
  for (int cell = tid; cell < Gm::cells; cell += blockDim.x) {
    const int a = cell / TW, b = cell % TW;
    const int u = u0 - R + a, v = v0 - R + b;
    float r = 0.f;
    if (u >= 0 && u < gh && v >= 0 && v < gw) {
      const uint8_t* p0 = keys + (size_t)cell * Gm::stride;
      float sn = 0.f;
#pragma unroll 4
      for (int c = 0; c < kChunks; ++c) {
        float x[kPer];
        unpack16<T>(*reinterpret_cast<const uint4*>(p0 + 16 * c), x);
#pragma unroll
        for (int t = 0; t < kPer; ++t) sn = fmaf(x[t], x[t], sn);
      }
      r = 1.0f / fmaxf(sqrtf(sn), 1e-8f);
      if (a >= R && a < R + kBoxRows && b >= R && b < R + kBoxCols) {
        const int j = off + u * gw + v;
        norms.rn.at(l)[(size_t)h * n + j] = r;
        if (norms.rho_key.base) norms.rho_key.at(l)[(size_t)h * n + j] = 0u;
        if (f == ft.n_frames - 1) norms.rn_cur.at(l)[(size_t)h * norms.cur_pad + (j - off)] = r;
      }
    }
    rn[cell] = r;
  }
  __syncthreads();
  // box sums: kLanes lanes = a pair of output columns
  constexpr int kPairs = kD / kLanes / 2;  // a lane's dimensions, in pairs
  const int dg = tid % kLanes, col = 2 * (tid / kLanes);
  float* phi = phi_all.at(l);
  auto load = [&](int cell, uint64_t (&x)[kPairs]) {
    const uint8_t* p0 = keys + (size_t)cell * Gm::stride + dg * kPairs * 2 * (int)sizeof(T);
    if constexpr (kPairs * 2 * sizeof(T) == 8) {  // 4 bf16
      const uint2 w = *reinterpret_cast<const uint2*>(p0);
      x[0] = pack_f2(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u));
      x[1] = pack_f2(__uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
    } else {
      float y[kPer];
      unpack16<T>(*reinterpret_cast<const uint4*>(p0), y);
#pragma unroll
      for (int t = 0; t < kPairs; ++t) x[t] = pack_f2(y[2 * t], y[2 * t + 1]);
    }
  };
  uint64_t ring[D2][2][kPairs];  // the last 2R+1 row sums of the two columns
#pragma unroll
  for (int a = 0; a < TH; ++a) {
    uint64_t(&hs)[2][kPairs] = ring[a % D2];
#pragma unroll
    for (int e = 0; e < kPairs; ++e) hs[0][e] = hs[1][e] = 0ull;
#pragma unroll
    for (int dv = 0; dv <= D2; ++dv) {
      const int cell = a * TW + col + dv;
      const float r = rn[cell];
      const uint64_t rr = pack_f2(r, r);
      uint64_t x[kPairs];
      load(cell, x);
#pragma unroll
      for (int e = 0; e < kPairs; ++e) {
        if (dv < D2) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(hs[0][e]) : "l"(rr), "l"(x[e]));
        if (dv > 0) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(hs[1][e]) : "l"(rr), "l"(x[e]));
      }
    }
    if (a >= 2 * R) {
      const int o = a - 2 * R;  // output row of the tile
      float dot[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int cell = (o + R) * TW + col + c + R;
        const float nr = -rn[cell];
        const uint64_t rr = pack_f2(nr, nr);
        uint64_t x[kPairs];
        load(cell, x);
        dot[c] = 0.f;
#pragma unroll
        for (int e = 0; e < kPairs; ++e) {
          uint64_t s = ring[0][c][e], nk;  // nk = -khat
#pragma unroll
          for (int q = 1; q < D2; ++q) asm("add.rn.f32x2 %0, %0, %1;" : "+l"(s) : "l"(ring[q][c][e]));
          asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(nk) : "l"(rr), "l"(x[e]));
          asm("add.rn.f32x2 %0, %0, %1;" : "+l"(s) : "l"(nk));
          const float2 sf = unpack_f2(s), kf = unpack_f2(nk);
          dot[c] = fmaf(-kf.x, sf.x, dot[c]);
          dot[c] = fmaf(-kf.y, sf.y, dot[c]);
        }
      }
      // the lower half of the lanes goes on with the first column, the upper half with the second
      const bool up = dg & (kLanes / 2);
      float d = (up ? dot[1] : dot[0]) + __shfl_xor_sync(0xffffffffu, up ? dot[0] : dot[1], kLanes / 2);
#pragma unroll
      for (int m = kLanes / 4; m > 0; m >>= 1) d += __shfl_xor_sync(0xffffffffu, d, m);
      const int u = u0 + o, v = v0 + col + (up ? 1 : 0);
      if (dg % (kLanes / 2) == 0 && u < gh && v < gw) {
        const int nu = min(u + R, gh - 1) - max(u - R, 0) + 1;
        const int nv = min(v + R, gw - 1) - max(v - R, 0) + 1;
        const int cnt = nu * nv - 1;
        phi[(size_t)h * n + off + u * gw + v] = cnt ? 1.0f - d / (float)cnt : 0.0f;
      }
    }
  }
}

template <typename T, int R>
static cudaError_t css_box_t(const Problem& p, const FrameTable& ft, const LayerPtrs& io, Strided<float> phi,
                             const NormsOut& norms, cudaStream_t st) {
  using Gm = BoxGeom<T, R>;
  cudaError_t e = cudaFuncSetAttribute(k_css_box<T, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, Gm::smem);
  if (e != cudaSuccess) return e;
  int tiles = 1;
  for (int f = 0; f < ft.n_frames; ++f) {
    const int t = ((ft.gh[f] + kBoxRows - 1) / kBoxRows) * ((ft.gw[f] + kBoxCols - 1) / kBoxCols);
    tiles = t > tiles ? t : tiles;
  }
  TimingScope ts("css_box", st);
  dim3 grid((unsigned)tiles, (unsigned)(ft.n_frames > 0 ? ft.n_frames : 1), (unsigned)(p.L * p.hkv));
  k_css_box<T, R><<<grid, Gm::threads, Gm::smem, st>>>(io, ft, p.hkv, phi, norms);
  return cudaGetLastError();
}

template <typename T>
static cudaError_t css_box_r(int radius, const Problem& p, const FrameTable& ft, const LayerPtrs& io,
                             Strided<float> phi, const NormsOut& norms, cudaStream_t st) {
  switch (radius) {
    case 1: return css_box_t<T, 1>(p, ft, io, phi, norms, st);
    case 2: return css_box_t<T, 2>(p, ft, io, phi, norms, st);
    case 3: return css_box_t<T, 3>(p, ft, io, phi, norms, st);
    case 4: return css_box_t<T, 4>(p, ft, io, phi, norms, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_css_box(const Problem& p, const FrameTable& ft, const LayerPtrs& io, int size,
                           Strided<float> phi, const NormsOut& norms, cudaStream_t st) {
  if (ft.n_frames == 0) return cudaSuccess;
  if (p.dtype == kBF16) return css_box_r<__nv_bfloat16>(size / 2, p, ft, io, phi, norms, st);
  return css_box_r<float>(size / 2, p, ft, io, phi, norms, st);
}

cudaError_t launch_fill_text_nan(const Problem& p, const FrameTable& ft, float* phi, cudaStream_t st) {
  long long tot = (long long)p.n * p.hkv;
  long long blocks = (tot + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  k_fill_text_nan<<<(int)blocks, 256, 0, st>>>(ft, p.hkv, phi);
  return cudaGetLastError();
}

// ------------------------------------------------------- row statistics
// Window score, first pass (fp32): for every query row r of KV head h (r =
// window row * G + group member) the maximum m and sum l of 2^(x - m), x =
// q.k * log2(e)/sqrt(d), over the keys of one split (whole 64-key tiles, so
// that the last splits may be empty).  A thread keeps its eight rows' states
// over the keys it sees; the sixteen threads of a row merge theirs at the
// end.  grid = (split, layer*Hkv + head, 64 query rows).
constexpr int kScoreSimtSmem = 2 * kTileFloats * 4;

// Query row r of KV head h.
__device__ __forceinline__ const float* q_row(const float* q, const Problem& p, int h, int r) {
  const int G = p.G(), wr = r / G;
  return q + ((size_t)wr * p.hq + h * G + (r - wr * G)) * kD;
}

__global__ void __launch_bounds__(kTileThreads, kTilesPerSm)
    k_rowstats_simt(const __grid_constant__ LayerPtrs io, Problem p, int nsplit, Strided<float2> part_all) {
  extern __shared__ float4 tile_smem[];
  float* qs = reinterpret_cast<float*>(tile_smem);
  float* ks = qs + kTileFloats;
  const int s = blockIdx.x, l = blockIdx.y / p.hkv, h = blockIdx.y % p.hkv, r0 = blockIdx.z * kTileRows;
  const float* q = static_cast<const float*>(io.q[l]);
  const float* k = static_cast<const float*>(io.k[l]);
  float2* part = part_all.at(l);
  const int R = p.R(), ty = tile_ty(), tx = tile_tx();
  const float c = kLog2e * rsqrtf((float)kD);
  const int per = ((p.n + nsplit - 1) / nsplit + kTileRows - 1) / kTileRows * kTileRows;
  const int j0 = min(p.n, s * per), j1 = min(p.n, j0 + per);
  tile_load(qs, min(kTileRows, R - r0), [&](int r) { return q_row(q, p, h, r0 + r); });
  float m[kTA], ls[kTA];
#pragma unroll
  for (int i = 0; i < kTA; ++i) {
    m[i] = -CUDART_INF_F;
    ls[i] = 0.f;
  }
  for (int jt = j0; jt < j1; jt += kTileRows) {
    const int nk = min(kTileRows, j1 - jt);
    tile_load(ks, nk, [&](int r) { return k + ((size_t)(jt + r) * p.hkv + h) * kD; });
    tile_ready();
    float d[kTA][kTB];
    tile_dots(qs, ks, d);
#pragma unroll
    for (int i = 0; i < kTA; ++i) {
#pragma unroll
      for (int j = 0; j < kTB; ++j) d[i][j] = tx + 16 * j < nk ? d[i][j] * c : -CUDART_INF_F;
      fold_scores(m[i], ls[i], d[i]);
    }
    __syncthreads();  // the key tile is rewritten
  }
  merge_rows(m, ls, ks);
  if (tx == 0)
#pragma unroll
    for (int i = 0; i < kTA; ++i) {
      const int row = r0 + ty + 8 * i;
      if (row < R) part[((size_t)h * nsplit + s) * R + row] = make_float2(m[i], ls[i]);
    }
}

// Merge the splits: bias[h][r] = -m_r - log2(G * l_r), so that 2^(x + bias) =
// softmax probability / G.
// Four lanes per query row (row_bias4).  grid.y = layer.
__global__ void __launch_bounds__(128) k_row_bias(Problem p, int nsplit, Strided<float2> part_all) {
  pdl_trigger();
  pdl_wait();
  const int R = p.R(), l = blockIdx.y;
  const float2* part = part_all.at(l);
  float* bias = reinterpret_cast<float*>(part_all.at(l) + (size_t)p.hkv * nsplit * R);
  const int e4 = blockIdx.x * blockDim.x + threadIdx.x, e = e4 >> 2;
  const bool live = e < p.hkv * R;
  const int h = live ? e / R : 0, r = live ? e - h * R : 0;
  const float v = row_bias4(part + (size_t)h * nsplit * R + r, R, live ? nsplit : 0, (float)p.G());
  if (live && (e4 & 3) == 0) bias[e] = v;
}

cudaError_t launch_row_bias(const Problem& p, int nsplit, Strided<float2> rowpart, cudaStream_t st) {
  const int rows = p.hkv * p.R();
  const cudaError_t e = launch_after(k_row_bias, dim3((4 * rows + 127) / 128, p.L), 128, 0, st, p, nsplit, rowpart);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// ---------------------------------------------------------- column sums
// Window score, second pass (fp32): a[h][j] = sum_r 2^(x_rj + bias_r).  The
// key tile stays, the query rows stream; a thread sums its eight keys over
// the rows it sees, the sixteen threads of a key add theirs at the end.  A
// cluster of CTAs may share a key tile: each takes every split-th tile of
// query rows, and their sums are added in rank order.
// grid = (key tile * split, layer*Hkv + head).
__global__ void __launch_bounds__(kTileThreads, kTilesPerSm)
    k_colsum_simt(const __grid_constant__ LayerPtrs io, Problem p, int nsplit, Strided<float2> part_all,
                  Strided<float> a_all) {
  extern __shared__ float4 tile_smem[];
  float* ks = reinterpret_cast<float*>(tile_smem);
  float* qs = ks + kTileFloats;
  cg::cluster_group cl = cg::this_cluster();
  const int split = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int l = blockIdx.y / p.hkv, h = blockIdx.y % p.hkv, j0 = (int)blockIdx.x / split * kTileRows;
  const float* q = static_cast<const float*>(io.q[l]);
  const float* k = static_cast<const float*>(io.k[l]);
  const int R = p.R(), ty = tile_ty(), tx = tile_tx();
  const float* bias = reinterpret_cast<const float*>(part_all.at(l) + (size_t)p.hkv * nsplit * R) + (size_t)h * R;
  const float c = kLog2e * rsqrtf((float)kD);
  tile_load(ks, min(kTileRows, p.n - j0), [&](int r) { return k + ((size_t)(j0 + r) * p.hkv + h) * kD; });
  float2 acc[kTA];
#pragma unroll
  for (int i = 0; i < kTA; ++i) acc[i] = make_float2(0.f, 0.f);
  for (int rt = rank * kTileRows; rt < R; rt += split * kTileRows) {
    const int nr = min(kTileRows, R - rt);
    tile_load(qs, nr, [&](int r) { return q_row(q, p, h, rt + r); });
    float bs[kTB];
#pragma unroll
    for (int j = 0; j < kTB; ++j) bs[j] = tx + 16 * j < nr ? __ldg(bias + rt + tx + 16 * j) : 0.f;
    tile_ready();
    float d[kTA][kTB];
    tile_dots(ks, qs, d);
#pragma unroll
    for (int i = 0; i < kTA; ++i) {
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < kTB; ++j) sum += tx + 16 * j < nr ? exp2f(fmaf(d[i][j], c, bs[j])) : 0.f;
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
  if (rank == 0 && threadIdx.x < kTileRows && j < p.n) {
    float2 total = sums[threadIdx.x];
    for (int r = 1; r < split; ++r) add_exact(total, cl.map_shared_rank(sums, r)[threadIdx.x]);
    a_all.at(l)[(size_t)h * p.n + j] = total.x + total.y;
  }
  if (split > 1) cl.sync();  // no CTA leaves while rank 0 may still read its sums
}

// CTAs per key tile: as many as there are tiles of query rows, while those of
// one layer all fit at once (1,152 keys of 4 heads: 72 key tiles for 456
// places; one CTA each worked off four tiles of query rows alone on its SM).
// It fixes how the sums are grouped, so it depends on the layer's shape alone.
static int colsum_simt_split(const Problem& p) {
  const long long tiles = (long long)((p.n + kTileRows - 1) / kTileRows) * p.hkv;
  const int rows = (p.R() + kTileRows - 1) / kTileRows;
  int s = 1;
  while (2 * s <= rows && 2 * s <= 8 && tiles * 2 * s <= 152 * kTilesPerSm) s *= 2;
  return s;
}

cudaError_t launch_score(const Problem& p, const LayerPtrs& io, Strided<float2> rowpart, int nsplit,
                         Strided<float> a_base, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(k_rowstats_simt, cudaFuncAttributeMaxDynamicSharedMemorySize, kScoreSimtSmem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_colsum_simt, cudaFuncAttributeMaxDynamicSharedMemorySize, kScoreSimtSmem);
  if (e != cudaSuccess) return e;
  dim3 g1(nsplit, p.L * p.hkv, (p.R() + kTileRows - 1) / kTileRows);
  const int split = colsum_simt_split(p);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3((p.n + kTileRows - 1) / kTileRows * split, p.L * p.hkv);
  cfg.blockDim = dim3(kTileThreads);
  cfg.dynamicSmemBytes = kScoreSimtSmem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)split;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  {
    TimingScope ts("rowstats_simt", st);
    k_rowstats_simt<<<g1, kTileThreads, kScoreSimtSmem, st>>>(io, p, nsplit, rowpart);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  {
    TimingScope ts("row_bias", st);
    if ((e = launch_row_bias(p, nsplit, rowpart, st)) != cudaSuccess) return e;
  }
  TimingScope ts("colsum_simt", st);
  e = cudaLaunchKernelEx(&cfg, k_colsum_simt, io, p, nsplit, rowpart, a_base);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// ------------------------------------------------------------------ TSG
// fp32 path of Eq. 6: a tile of 64 historical tokens against the current
// frame's keys of one column slice, streamed in tiles of 64; the slices fold
// into rho_key.  grid = (half row tile, layer*Hkv + head, slice).
constexpr int kTsgSimtSmem = (2 * kTileFloats + 2 * kTileRows) * 4;

__global__ void __launch_bounds__(kTileThreads, kTilesPerSm)
    k_tsg_simt(const __grid_constant__ LayerPtrs io, const __grid_constant__ FrameTable ft, int hkv,
               Strided<const float> rn_all, Strided<uint32_t> rho_all, int slice_cols, int metric) {
  extern __shared__ float4 tile_smem[];
  float* hs = reinterpret_cast<float*>(tile_smem);
  float* cs = hs + kTileFloats;
  float* cr = cs + kTileFloats;  // [64] scale of each current key
  float* co = cr + kTileRows;    // [64] offset: value = dot * scale + offset
  const int t = blockIdx.x >> 1, l = blockIdx.y / hkv, h = blockIdx.y % hkv, tid = threadIdx.x;
  const int n = ft.n_tokens, ty = tile_ty(), tx = tile_tx();
  const float* k = static_cast<const float*>(io.k[l]);
  const float* rn = rn_all.at(l) + (size_t)h * n + ft.cur_off;
  // tile -> historical frame
  int f = 0;
  while (f + 1 < ft.n_frames - 1 && ft.tile0[f + 1] <= t) ++f;
  const int fend = ft.off[f] + ft.gh[f] * ft.gw[f];
  const int i0 = ft.off[f] + (t - ft.tile0[f]) * kTsgTile + (blockIdx.x & 1) * kTileRows;
  if (i0 >= fend) return;  // the frame's last 128-token tile is at most half full
  auto key_row = [&](int j) { return k + ((size_t)j * hkv + h) * kD; };
  tile_load(hs, min(kTileRows, fend - i0), [&](int r) { return key_row(i0 + r); });
  float best[kTA];
#pragma unroll
  for (int i = 0; i < kTA; ++i) best[i] = -CUDART_INF_F;
  const int jend = min(ft.cur_len, (int)(blockIdx.z + 1) * slice_cols);
  for (int jt = blockIdx.z * slice_cols; jt < jend; jt += kTileRows) {
    const int nk = min(kTileRows, jend - jt);
    tile_load(cs, nk, [&](int r) { return key_row(ft.cur_off + jt + r); });
    if (tid < kTileRows) {
      // cosine: dot * rn_j; dot: dot; negative L2 (without the row's own
      // -|k_i|^2): 2 dot - |k_j|^2; columns past the slice lose every maximum
      const float r = tid < nk ? rn[jt + tid] : 0.f;
      cr[tid] = metric == kTsgCosine ? r : (metric == kTsgDot ? 1.f : 2.f);
      co[tid] = tid >= nk ? -CUDART_INF_F : (metric == kTsgNegL2 ? -1.f / (r * r) : 0.f);
    }
    tile_ready();
    float d[kTA][kTB];
    tile_dots(hs, cs, d);
#pragma unroll
    for (int j = 0; j < kTB; ++j) {
      const float a = cr[tx + 16 * j], b = co[tx + 16 * j];
#pragma unroll
      for (int i = 0; i < kTA; ++i) best[i] = fmaxf(best[i], fmaf(d[i][j], a, b));
    }
    __syncthreads();  // the column tile is rewritten
  }
#pragma unroll
  for (int i = 0; i < kTA; ++i)
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) best[i] = fmaxf(best[i], __shfl_xor_sync(0xffffffffu, best[i], o));
  if (tx == 8)
#pragma unroll
    for (int i = 0; i < kTA; ++i) cs[ty + 8 * i] = best[i];
  __syncthreads();
  uint32_t* rho_key = rho_all.at(l) + (size_t)h * n;
  if (tx == 0)
#pragma unroll
    for (int i = 0; i < kTA; ++i) {
      const int tok = i0 + ty + 8 * i;
      if (tok < fend) atomicMax(rho_key + tok, float_key(fmaxf(best[i], cs[ty + 8 * i])));
    }
}

// Column slices of the fp32 TSG pass: the count whose CTAs, three to an SM,
// take the least time in whole waves, a wave costing its column tiles plus
// about one for the row tile's load.  The slices fold by maximum, so the
// count changes no result.
static int tsg_simt_slices(const Problem& p, const FrameTable& ft) {
  const long long rows = 2LL * ft.tile0[ft.n_frames - 1] * p.L * p.hkv;
  const int tiles = (ft.cur_len + kTileRows - 1) / kTileRows;
  const long long slots = 152 * kTilesPerSm;
  int best = 1;
  long long best_cost = 0;
  for (int s = 1; s <= tiles && s <= 16; ++s) {
    const int per = (tiles + s - 1) / s;
    if ((s - 1) * per >= tiles) continue;  // an empty slice
    const long long cost = ((rows * s + slots - 1) / slots) * (per + 1);
    if (s == 1 || cost < best_cost) {
      best = s;
      best_cost = cost;
    }
  }
  return best;
}

cudaError_t launch_tsg(const Problem& p, const FrameTable& ft, const LayerPtrs& io, Strided<const float> rn,
                       Strided<uint32_t> rho_key, int metric, cudaStream_t st) {
  const int tiles = ft.n_frames >= 2 ? ft.tile0[ft.n_frames - 1] : 0;
  if (tiles == 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_tsg_simt, cudaFuncAttributeMaxDynamicSharedMemorySize, kTsgSimtSmem);
  if (e != cudaSuccess) return e;
  const int slices = tsg_simt_slices(p, ft);
  const int ctiles = (ft.cur_len + kTileRows - 1) / kTileRows;
  const int slice_cols = (ctiles + slices - 1) / slices * kTileRows;
  TimingScope ts("tsg_simt", st);
  k_tsg_simt<<<dim3(2 * tiles, p.L * p.hkv, slices), kTileThreads, kTsgSimtSmem, st>>>(io, ft, p.hkv, rn, rho_key,
                                                                                      slice_cols, metric);
  return cudaGetLastError();
}

}  // namespace stl
