// Activation transform + block clip + MXFP4 / MXFP8 quantiser (stages 1+2 of the path) for some dozens
// of tokens: one thread per (token, block), a warp takes 32 tokens of ONE block.
//
// The per-block kernel (four lanes per item) loads its factors anew for every item, 256 bytes of L1
// traffic per lane, which is what bounds it from some 8000 items on.  Here the factors of a warp are the
// same in all lanes (broadcast loads, once per CTA), the Kronecker form runs as packed fp32 FMAs, and
// there is no shared memory and no barrier.  The same fused multiply-adds in the same order as the other
// ALU kernels: identical codes.  440 instructions per 32 items; a launch of one tile per CTA is a chain
// of latencies (factors, wait, X, 440 instructions, stores).
// Measured back to back, this / per-block kernel: 4096 channels, 75 tokens 2.6 / 3.1 us, 128 tokens
// 2.6 / 3.6; 14336 channels, 75 tokens 3.6 / 5.2, 128 tokens 4.2 / 8.0.
#pragma once
#include "ptx.cuh"
#include "quantize_act.cuh"
#include "quantize_act_tc.cuh"

namespace batq {

constexpr int kQwThreads = 128;   // 4 warps = the 4 blocks of one scale atom
constexpr int kQwRows = 32;       // tokens of a warp at a time

struct QuantWarpParams {
  const uint16_t* x;     // bf16 bits [s x n], row stride ld
  int64_t ld;
  int64_t s;
  int32_t n;
  int32_t k;             // n / 32
  int32_t n_tiles;       // 32-token tiles
  int32_t tiles_per_cta; // consecutive ones, grid.y CTAs per 4 blocks
  const float* left;     // [.][gr x gr], left_stride floats apart (0 = shared)
  const float* right;    // [.][gc x gc]
  int32_t left_stride;
  int32_t right_stride;
  const float* clip_lo;  // [k] or NULL
  const float* clip_hi;
  uint8_t* codes;        // [s x n/2], FP8: [s x n]
  uint8_t* scales;
  int32_t sf_layout;     // BATQ_SF_ROWMAJOR / BATQ_SF_MMA
  int32_t sf_katoms;
  uint32_t* zero_words;  // optional: n_zero_words 32-bit words set to zero (tickets of the kernel that follows)
  int32_t n_zero_words;
};

// Two fp32 values in one 64-bit register pair; both halves round as the scalar operation does.
__device__ __forceinline__ uint64_t f32x2_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f32x2_unpack(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t f32x2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f32x2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// GC = size of the right factor (8 or 4; the left one is 32 / GC).
template <int GC, bool CLIP, bool FP8>
__global__ void __launch_bounds__(kQwThreads, 3) quantize_act_warp_kernel(const QuantWarpParams p) {
  constexpr int GR = 32 / GC, CP = GC / 2;
  grid_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j = static_cast<int>(blockIdx.x) * 4 + warp;
  const int t0 = static_cast<int>(blockIdx.y) * p.tiles_per_cta;
  const int t1 = min(p.n_tiles, t0 + p.tiles_per_cta);
  auto clear = [&] {   // by all warps of CTA (0, 0), those of padding blocks too
    if (blockIdx.x == 0 && blockIdx.y == 0)
      for (int i = threadIdx.x; i < p.n_zero_words; i += kQwThreads) p.zero_words[i] = 0u;
  };
  if (j >= p.k) {   // padding blocks of the scale layout: keep them finite
    grid_dependency_wait();
    clear();
    if (p.sf_layout != 0)
      for (int t = t0; t < t1; ++t) {
        const int64_t row = static_cast<int64_t>(t) * kQwRows + lane;
        if (row < p.s) p.scales[sf_mma_offset(row, j, p.sf_katoms)] = 0;
      }
    return;
  }
  uint64_t R[GC][CP];   // pairs of neighbouring columns
  {
    const ulonglong2* rp = reinterpret_cast<const ulonglong2*>(p.right + static_cast<int64_t>(j) * p.right_stride);
#pragma unroll
    for (int i = 0; i < GC * CP / 2; ++i) {
      const ulonglong2 v = __ldg(rp + i);
      R[2 * i / CP][2 * i % CP] = v.x;
      R[(2 * i + 1) / CP][(2 * i + 1) % CP] = v.y;
    }
  }
  float L[GR][GR];
  {
    const float4* lp = reinterpret_cast<const float4*>(p.left + static_cast<int64_t>(j) * p.left_stride);
#pragma unroll
    for (int i = 0; i < GR * GR / 4; ++i) {
      const float4 v = __ldg(lp + i);
      float* d = &L[0][0] + 4 * i;
      d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
    }
  }
  float c_lo = 1.0f, c_hi = 1.0f;
  if (CLIP) { c_lo = __ldg(p.clip_lo + j); c_hi = __ldg(p.clip_hi + j); }
  // x may come from the grid in front, which may also still read the codes, scales and tickets of its own call
  grid_dependency_wait();
  clear();
  const uint16_t* xj = p.x + static_cast<int64_t>(j) * 32;
  uint4 x[4];
  auto load = [&](int t) {
    const int64_t row = static_cast<int64_t>(t) * kQwRows + lane;
    const bool in = t < t1 && row < p.s;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[i] = make_uint4(0u, 0u, 0u, 0u);
      if (in) x[i] = ld_global_ordered_v4(xj + row * p.ld + 8 * i);
    }
  };
  load(t0);
#pragma unroll 1
  for (int tile = t0; tile < t1; ++tile) {
    const int64_t row = static_cast<int64_t>(tile) * kQwRows + lane;
    uint64_t U[GR][CP];   // V R
#pragma unroll
    for (int r = 0; r < GR; ++r)
#pragma unroll
      for (int cc = 0; cc < GC; ++cc) {
        const int e = r * GC + cc;
        const uint4& q = x[e >> 3];
        const uint32_t w = (e & 7) < 2 ? q.x : (e & 7) < 4 ? q.y : (e & 7) < 6 ? q.z : q.w;
        const float v = __uint_as_float((e & 1) ? (w & 0xFFFF0000u) : (w << 16));
        const uint64_t vv = f32x2_pack(v, v);
#pragma unroll
        for (int c = 0; c < CP; ++c) U[r][c] = cc == 0 ? f32x2_mul(vv, R[0][c]) : f32x2_fma(vv, R[cc][c], U[r][c]);
      }
    load(tile + 1);
    float o[32];          // L^T (V R)
#pragma unroll
    for (int r = 0; r < GR; ++r) {
      uint64_t a[CP];
#pragma unroll
      for (int i = 0; i < GR; ++i) {
        const uint64_t ll = f32x2_pack(L[i][r], L[i][r]);
#pragma unroll
        for (int c = 0; c < CP; ++c) a[c] = i == 0 ? f32x2_mul(ll, U[0][c]) : f32x2_fma(ll, U[i][c], a[c]);
      }
#pragma unroll
      for (int c = 0; c < CP; ++c) f32x2_unpack(a[c], o[r * GC + 2 * c], o[r * GC + 2 * c + 1]);
    }
    float mn[4], mx[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      mn[i] = fmin3(fmin3(o[i], o[i + 4], o[i + 8]), fmin3(o[i + 12], o[i + 16], o[i + 20]), fminf(o[i + 24], o[i + 28]));
      mx[i] = fmax3(fmax3(o[i], o[i + 4], o[i + 8]), fmax3(o[i + 12], o[i + 16], o[i + 20]), fmaxf(o[i + 24], o[i + 28]));
    }
    const float mnv = fminf(fmin3(mn[0], mn[1], mn[2]), mn[3]), mxv = fmaxf(fmax3(mx[0], mx[1], mx[2]), mx[3]);
    float amax;
    if (CLIP) {
      const float lo = c_lo * mnv, hi = c_hi * mxv;
#pragma unroll
      for (int i = 0; i < 32; ++i) o[i] = fminf(fmaxf(o[i], lo), hi);
      amax = fmaxf(fabsf(fminf(fmaxf(mnv, lo), hi)), fabsf(fminf(fmaxf(mxv, lo), hi)));
    } else {
      amax = fmaxf(fabsf(mnv), fabsf(mxv));
    }
    // shared scale: byte = max(biased_exponent(amax) - emax, 0), emax = 2 (E2M1) or 8 (E4M3)
    const int ef = static_cast<int>(__float_as_uint(amax) >> 23);
    const int sbyte = max(ef - (FP8 ? 8 : 2), 0);
    const float inv = __uint_as_float(static_cast<uint32_t>(254 - sbyte) << 23);
#pragma unroll
    for (int i = 0; i < 32; i += 2) mul2(o[i], o[i + 1], inv, o[i], o[i + 1]);
    if (row >= p.s) continue;
    if (FP8) {
      uint4* dst = reinterpret_cast<uint4*>(p.codes + row * p.n + static_cast<int64_t>(j) * 32);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t cw[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          cw[i] = e4m3x4_pack(o[16 * h + 4 * i], o[16 * h + 4 * i + 1], o[16 * h + 4 * i + 2], o[16 * h + 4 * i + 3]);
        dst[h] = make_uint4(cw[0], cw[1], cw[2], cw[3]);
      }
    } else {
      uint32_t cw[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float uu[8] = {o[8 * i], o[8 * i + 1], o[8 * i + 2], o[8 * i + 3], o[8 * i + 4], o[8 * i + 5], o[8 * i + 6], o[8 * i + 7]};
        cw[i] = e2m1x8_pack(uu);
      }
      *reinterpret_cast<uint4*>(p.codes + row * (p.n / 2) + static_cast<int64_t>(j) * 16) = make_uint4(cw[0], cw[1], cw[2], cw[3]);
    }
    if (p.sf_layout == 0) p.scales[row * p.k + j] = static_cast<uint8_t>(sbyte);
    else p.scales[sf_mma_offset(row, j, p.sf_katoms)] = static_cast<uint8_t>(sbyte);
  }
}

}  // namespace batq
