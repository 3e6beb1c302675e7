// Building blocks of the fp32 kernels (intra_simt.cu, chain_simt.cu, bwd_exact.cu): register-tiled fp32 products on
// shared memory, and the tile loads in front of them.
//
// Why packed FMAs and k-contiguous operands: these kernels are bound by the fp32 FMA pipes and the shared-memory port.
// Both operands of a product are kept with the summed index contiguous, so that one 16-byte load brings four terms of
// a row, and a pair of terms is one two-lane FMA (__ffma2_rn) without any register shuffling; the two lanes of an
// accumulator hold the even and the odd terms and are added at the end.  Rows are padded by four floats: eight
// consecutive rows (or columns) then lie in different 16-byte bank groups, so a warp's loads (8 x 4 distinct rows) take
// one wavefront each.
#pragma once
#include "mdn_common.cuh"

namespace mdn {

constexpr int kSimtThreads = 256;
constexpr int kLT = C + 4;   // floats per row of a 64-wide matrix

__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void fma4(float2& acc, const float4& a, const float4& b) {
  acc = __ffma2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y), acc);
  acc = __ffma2_rn(make_float2(a.z, a.w), make_float2(b.z, b.w), acc);
}
__device__ __forceinline__ float hsum(const float2& x) { return x.x + x.y; }

template <int R, int N> __device__ __forceinline__ void zero2(float2 (&acc)[R][N]) {
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) acc[i][j] = make_float2(0.f, 0.f);
}

// acc[i][j] += sum over 4 k0 <= k < 4 k1 of a[i * a_step + k] * b[j * b_step + k]
template <int R, int N>
__device__ __forceinline__ void dot_tile(float2 (&acc)[R][N], const float* a, int a_step, const float* b, int b_step, int k0,
                                         int k1) {
#pragma unroll 2
  for (int k = k0; k < k1; ++k) {
    float4 av[R], bv[N];
#pragma unroll
    for (int i = 0; i < R; ++i) av[i] = lds4(a + i * a_step + 4 * k);
#pragma unroll
    for (int j = 0; j < N; ++j) bv[j] = lds4(b + j * b_step + 4 * k);
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < N; ++j) fma4(acc[i][j], av[i], bv[j]);
  }
}

// ---- asynchronous loads (cp.async, 16 bytes; dead pieces are zero-filled)
__device__ __forceinline__ void cp16(void* dst, const void* src, bool live) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(live ? 16 : 0));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// 64 rows of D values (row_stride elements apart, rows >= n zero): fp32 input goes straight into the padded tile, bf16
// input into `raw` (64 x D bf16), from which widen_tile fills the tile after the copy has landed.
template <int D>
__device__ __forceinline__ void load_rows(float* tile, void* raw, const void* src, bool bf16, size_t row_stride, int n, int tid) {
  if (!bf16) {
    for (int i = tid; i < C * (D / 4); i += kSimtThreads) {
      const int r = i / (D / 4), c = (i % (D / 4)) * 4;
      cp16(tile + r * (D + 4) + c, static_cast<const float*>(src) + (r < n ? r : 0) * row_stride + c, r < n);
    }
  } else {
    for (int i = tid; i < C * (D / 8); i += kSimtThreads) {
      const int r = i / (D / 8), c = (i % (D / 8)) * 8;
      cp16(static_cast<__nv_bfloat16*>(raw) + r * D + c, static_cast<const __nv_bfloat16*>(src) + (r < n ? r : 0) * row_stride + c,
           r < n);
    }
  }
}
template <int D> __device__ __forceinline__ void widen_tile(float* tile, const void* raw, int tid) {
  for (int i = tid; i < C * (D / 4); i += kSimtThreads) {
    const int r = i / (D / 4), c = (i % (D / 4)) * 4;
    const uint2 u = *reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(raw) + r * D + c);
    *reinterpret_cast<float4*>(tile + r * (D + 4) + c) =
        make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                    __uint_as_float(u.y & 0xffff0000u));
  }
}
// a 64 x 64 fp32 matrix (rows of 64) into a padded one
__device__ __forceinline__ void load_mat(float* dst, const float* src, int tid) {
  for (int i = tid; i < C * 16; i += kSimtThreads) cp16(dst + (i >> 4) * kLT + (i & 15) * 4, src + i * 4, true);
}

__device__ __forceinline__ float load_io(const void* p, size_t i, bool bf16) {
  return bf16 ? __bfloat162float(__ldg(static_cast<const __nv_bfloat16*>(p) + i)) : __ldg(static_cast<const float*>(p) + i);
}
__device__ __forceinline__ void store_io(void* p, size_t i, bool bf16, float x) {
  if (bf16) static_cast<__nv_bfloat16*>(p)[i] = __float2bfloat16_rn(x);
  else static_cast<float*>(p)[i] = x;
}

}  // namespace mdn
