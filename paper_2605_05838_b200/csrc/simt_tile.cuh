// Building blocks of the fp32 kernels (intra_simt.cu, chain_simt.cu, bwd_exact.cu): register-tiled fp32 products on
// shared memory, and the tile loads in front of them.
//
// What bounds them: the shared-memory port, before the fp32 pipes.  A 16-byte load returns 512 bytes to a warp and
// takes four cycles of the port whether its lanes' addresses repeat or not (measured: 11.6 k wavefronts per chunk where
// one per distinct 128 bytes would have been 3.6 k), so an R x N tile per thread costs 4 (R + N) port cycles per R N FMA-pipe cycles of
// its warp: only 8 x 8 is balanced.  Where a product has too few outputs to give every thread such a tile, the
// SUMMED index is split over SL neighbouring lanes (dot_slices / rank1 below), and the lanes' partial tiles are added by
// a shuffle reduction that leaves each lane 1 / SL of the sums (reduce_scatter).
// Both operands of a dot product are kept with the summed index contiguous: one 16-byte load brings four terms of a
// row, and a pair of terms is one two-lane FMA (__ffma2_rn, half the issue slots) without register shuffling.  Rows are padded by four floats, so that
// the eight lanes of a load phase (slices of a row, or rows four apart) fall into different bank groups.
#pragma once
#include "mdn_common.cuh"

namespace mdn {

constexpr int kSimtThreads = 256;
// The chain kernels take 16 threads per value column (128 or 256 per CTA): the tiles below then split every sum over
// the same number of lanes whatever NV is, so a result does not depend on the number of chains it was computed with.
template <int NV> constexpr int kChainThreads = 16 * NV;
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

// acc[i][j] += sum over the 4-term groups k0, k0 + step, .. < k1 of a_i[4 k ..] . b_j[4 k ..];  row i of A: a(i), column j of B: b(j)
template <int R, int N, class FA, class FB>
__device__ __forceinline__ void dot_slices(float2 (&acc)[R][N], FA a, FB b, int k0, int k1, int step) {
#pragma unroll 1
  for (int k = k0; k < k1; k += step) {
    float4 av[R], bv[N];
#pragma unroll
    for (int i = 0; i < R; ++i) av[i] = lds4(a(i) + 4 * k);
#pragma unroll
    for (int j = 0; j < N; ++j) bv[j] = lds4(b(j) + 4 * k);
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < N; ++j) fma4(acc[i][j], av[i], bv[j]);
  }
}

// Adds the SL lanes' (lane bits 0 .. log2 SL - 1) partial values v[0 .. CNT); afterwards v[0 .. CNT / SL) of the lane with
// slice s are the sums of elements s CNT / SL + (0 .. CNT / SL - 1).
template <int CNT, int SL> __device__ __forceinline__ void reduce_scatter(float (&v)[CNT], int s) {
  int cur = CNT;
#pragma unroll
  for (int off = SL / 2; off > 0; off >>= 1) {
    const bool up = (s & off) != 0;
    cur >>= 1;
#pragma unroll
    for (int i = 0; i < CNT / 2; ++i) {
      if (i < cur) {
        const float give = up ? v[i] : v[i + cur], keep = up ? v[i + cur] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
      }
    }
  }
}

// Rank-one updates acc[(8 key rows)][(4 columns)][2] += k_r (x) (w_r, w'_r) over the rows r = s, s + SL, .. < n of a tile:
// the thread's key rows are d0 .. d0 + 3 and d1 .. d1 + 3 of kt (row stride ldk), its columns four neighbouring ones of w
// ([r][column] pairs of weights, one per state; row stride ldw floats).
template <int SL>
__device__ __forceinline__ void rank1(float2 (&acc)[4][8], const float* kt, int ldk, int d0, int d1, const float* w, int ldw, int s, int n) {
#pragma unroll 2
  for (int r = s; r < n; r += SL) {
    const float4 ka = lds4(kt + r * ldk + d0), kb = lds4(kt + r * ldk + d1);
    const float4 wa = lds4(w + r * ldw), wb = lds4(w + r * ldw + 4);
    const float2 kv[4] = {make_float2(ka.x, ka.y), make_float2(ka.z, ka.w), make_float2(kb.x, kb.y), make_float2(kb.z, kb.w)};
    const float wv[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
    for (int c = 0; c < 8; ++c)
#pragma unroll
      for (int p = 0; p < 4; ++p) acc[p][c] = __ffma2_rn(kv[p], make_float2(wv[c], wv[c]), acc[p][c]);
  }
}

// ---- the tiles of the two chain kernels (NV value columns, dk = DK key rows)
// Products of 64-row tiles with both states: NA operands (K, or K and Q) x 8 / NA rows rt + (64 NA / 8) i, columns ct + (NV / 4) j
// of S and of M (j < 4).
template <int NV, int NA> struct StateTile {
  static constexpr int kRt = 8 * NA, kCt = NV / 4, SL = kChainThreads<NV> / (kRt * kCt), RI = 8 / NA;
  static_assert(SL == 4 || SL == 8 || SL == 16, "slices");
  int s, rt, ct;
  __device__ __forceinline__ StateTile(int tid) {
    const int t = tid / SL;
    s = tid % SL;
    ct = t / kRt;
    rt = t % kRt;
    if (SL == 4) rt = ((rt & 1) << 2) | ((rt >> 1) & 3) | (rt & 8);   // a phase's two tiles: rows four apart
  }
  static constexpr int kPairs = 32 / SL;   // (row, column) positions a lane ends up with
  // the lane's positions: f(n-th, which operand, row, column)
  template <class F> __device__ __forceinline__ void own(F f) const {
#pragma unroll
    for (int e = 0; e < kPairs; ++e) {
      const int idx = 2 * (s * kPairs + e), i = idx >> 3, j = (idx >> 1) & 3;
      f(e, i / RI, rt + kRt * (i % RI), ct + kCt * j);
    }
  }
  // sums over the key index; f(n-th, which operand, row, column, value against S, value against M)
  template <int DK, class F>
  __device__ __forceinline__ void run(const float* A0, const float* A1, const float* St, F f) const {
    constexpr int LDK = DK + 4;
    float2 acc[8][8];
    zero2(acc);
    const float* a0 = A0 + rt * LDK;
    const float* a1 = A1 + rt * LDK;
    const float* b0 = St + ct * LDK;
    dot_slices<8, 8>(acc, [&](int i) { return (i < RI ? a0 : a1) + (i % RI) * kRt * LDK; },
                     [&](int j) { return b0 + ((j >> 2) * NV + (j & 3) * kCt) * LDK; }, s, DK / 4, SL);
    float v[64];   // [operand][row][column][state]
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) { v[i * 8 + 2 * j] = hsum(acc[i][j]); v[i * 8 + 2 * j + 1] = hsum(acc[i][j + 4]); }
    reduce_scatter<64, SL>(v, s);
    own([&](int e, int which, int r, int j) { f(e, which, r, j, v[2 * e], v[2 * e + 1]); });
  }
};

// Products of a 64 x 64 triangular matrix with NV columns: 4 neighbouring rows x 4 columns ct + (NV / 4) j.
template <int NV> struct TriTile {
  static constexpr int kCt = NV / 4, SL = kChainThreads<NV> / (16 * kCt);
  int s, rt, ct;
  __device__ __forceinline__ TriTile(int tid) { const int t = tid / SL; s = tid % SL; rt = t % 16; ct = t / 16; }
  static constexpr int kOwn = 16 / SL;   // outputs a lane ends up with
  template <class F> __device__ __forceinline__ void own(F f) const {   // f(n-th, row, column)
#pragma unroll
    for (int e = 0; e < kOwn; ++e) {
      const int idx = s * kOwn + e;
      f(e, 4 * rt + (idx >> 2), ct + kCt * (idx & 3));
    }
  }
  // out[r][j] = sum_x A[r][x] B[j][x] over x <= r (lower) or x >= r (upper); f(row, column, value)
  template <bool kLower, class F> __device__ __forceinline__ void run(const float* A, const float* B, F f) const {
    float2 acc[4][4];
    zero2(acc);
    const float* a0 = A + 4 * rt * kLT;
    const float* b0 = B + ct * kLT;
    dot_slices<4, 4>(acc, [&](int i) { return a0 + i * kLT; }, [&](int j) { return b0 + j * kCt * kLT; },
                     kLower ? s : rt + s, kLower ? rt + 1 : 16, SL);
    float v[16];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) v[i * 4 + j] = hsum(acc[i][j]);
    reduce_scatter<16, SL>(v, s);
    own([&](int e, int r, int j) { f(r, j, v[e]); });
  }
};

// The rank-64 update of both states: key rows 4 dt .. + 3 and dk / 2 + 4 dt .. + 3, four neighbouring columns.
template <int DK, int NV> struct UpdateTile {
  static constexpr int kDt = DK / 8, kJt = NV / 4, SL = kChainThreads<NV> / (kDt * kJt), LDK = DK + 4, LDW = 2 * NV + 4;
  int s, dt, jt;
  float2 acc[4][8];
  __device__ __forceinline__ UpdateTile(int tid) {
    const int t = tid / SL;
    s = tid % SL;
    jt = t / kDt;
    dt = t % kDt;
    if (SL == 4) dt = ((dt & 1) << 2) | ((dt >> 1) & 3) | (dt & 8);
    zero2(acc);
  }
  __device__ __forceinline__ void add(const float* tile, const float* w, int n) {
    rank1<SL>(acc, tile, LDK, 4 * dt, DK / 2 + 4 * dt, w + 8 * jt, LDW, s, n);
  }
  // f(key row, column, sum for the first state, for the second)
  template <class F> __device__ __forceinline__ void finish(F f) {
    float v[64];   // [key row][column][state]
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int c = 0; c < 8; ++c) { v[(2 * p) * 8 + c] = acc[p][c].x; v[(2 * p + 1) * 8 + c] = acc[p][c].y; }
    reduce_scatter<64, SL>(v, s);
    constexpr int kOwn = 64 / SL;
#pragma unroll
    for (int e = 0; e < kOwn; e += 2) {
      const int idx = s * kOwn + e, i = idx >> 3, j = (idx >> 1) & 3;
      f((i >> 2) * (DK / 2) + 4 * dt + (i & 3), 4 * jt + j, v[e], v[e + 1]);
    }
  }
};

// ---- asynchronous loads (cp.async, 16 bytes; dead pieces are zero-filled)
__device__ __forceinline__ void cp16(void* dst, const void* src, bool live) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(live ? 16 : 0));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// 64 rows of D values (row_stride elements apart, rows >= n zero): fp32 input goes straight into the padded tile, bf16
// input into `raw` (64 x D bf16), from which widen_tile fills the tile after the copy has landed.
template <int D, int TH = kSimtThreads>
__device__ __forceinline__ void load_rows(float* tile, void* raw, const void* src, bool bf16, size_t row_stride, int n, int tid) {
  if (!bf16) {
    for (int i = tid; i < C * (D / 4); i += TH) {
      const int r = i / (D / 4), c = (i % (D / 4)) * 4;
      cp16(tile + r * (D + 4) + c, static_cast<const float*>(src) + (r < n ? r : 0) * row_stride + c, r < n);
    }
  } else {
    for (int i = tid; i < C * (D / 8); i += TH) {
      const int r = i / (D / 8), c = (i % (D / 8)) * 8;
      cp16(static_cast<__nv_bfloat16*>(raw) + r * D + c, static_cast<const __nv_bfloat16*>(src) + (r < n ? r : 0) * row_stride + c,
           r < n);
    }
  }
}
template <int D, int TH = kSimtThreads> __device__ __forceinline__ void widen_tile(float* tile, const void* raw, int tid) {
  for (int i = tid; i < C * (D / 4); i += TH) {
    const int r = i / (D / 4), c = (i % (D / 4)) * 4;
    const uint2 u = *reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(raw) + r * D + c);
    *reinterpret_cast<float4*>(tile + r * (D + 4) + c) =
        make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                    __uint_as_float(u.y & 0xffff0000u));
  }
}
// 64 rows of one head of an i/o tensor into a padded fp32 tile without staging (bf16: through registers, at once; fp32:
// asynchronously); src: the head's first element, rows row_stride elements apart.
__device__ __forceinline__ void load_io_rows(float* tile, const void* src, bool bf16, int D, size_t row_stride, int n, int tid) {
  if (!bf16) {
    const int per = D / 4;
    for (int i = tid; i < C * per; i += kSimtThreads) {
      const int r = i / per, c = (i % per) * 4;
      cp16(tile + r * (D + 4) + c, static_cast<const float*>(src) + (r < n ? r : 0) * row_stride + c, r < n);
    }
    return;
  }
  const int per = D / 8;
  for (int i = tid; i < C * per; i += kSimtThreads) {
    const int r = i / per, c = (i % per) * 8;
    uint4 u = make_uint4(0u, 0u, 0u, 0u);
    if (r < n) u = __ldg(reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(src) + r * row_stride + c));
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
    float f[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) { f[2 * e] = __uint_as_float(w[e] << 16); f[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u); }
    *reinterpret_cast<float4*>(tile + r * (D + 4) + c) = make_float4(f[0], f[1], f[2], f[3]);
    *reinterpret_cast<float4*>(tile + r * (D + 4) + c + 4) = make_float4(f[4], f[5], f[6], f[7]);
  }
}
// a 64 x 64 fp32 matrix (rows of 64) into a padded one
template <int TH>
__device__ __forceinline__ void load_mat(float* dst, const float* src, int tid) {
  for (int i = tid; i < C * 16; i += TH) cp16(dst + (i >> 4) * kLT + (i & 15) * 4, src + i * 4, true);
}

__device__ __forceinline__ float load_io(const void* p, size_t i, bool bf16) {
  return bf16 ? __bfloat162float(__ldg(static_cast<const __nv_bfloat16*>(p) + i)) : __ldg(static_cast<const float*>(p) + i);
}
__device__ __forceinline__ void store_io(void* p, size_t i, bool bf16, float x) {
  if (bf16) static_cast<__nv_bfloat16*>(p)[i] = __float2bfloat16_rn(x);
  else static_cast<float*>(p)[i] = x;
}

}  // namespace mdn
