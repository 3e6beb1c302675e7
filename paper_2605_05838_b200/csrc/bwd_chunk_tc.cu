// Chunk-parallel backward, stage 2 on the 5th-generation tensor cores: per (chunk, head), from the kept forward states
// (S, M at the chunk's start) and the adjoint pair (dS', dM' at its end), the gradients of q, k and of the four gates.
// Section 3.1-3.2: the chunk form in the notation of chain_tensor.cu,
//     X = K S,  Y = K M,  R = V - abar.X + p.Y,  V~ = T R,  T = (I + A)^-1,  A = G^- o (K K^T),  W = scale Geta o (Q K^T),
//     O = scale (abar.(Q S) - b.(Q M)) + W V~,   S' = abar_C S - b_C M + K^T (g_S.V~),   M' = mubar_C M - K^T (g_M.V~),
// differentiated matrix by matrix (dR = T^T dV~ = dV comes from the adjoint chain):
//     dQ  = scale (abar.(dO S^T) - b.(dO M^T)) + DW K,                    DW = scale Geta o tril(dO V~^T),
//     dK  = -abar.(dR S^T) + p.(dR M^T) + g_S.(V~ dS'^T) - g_M.(V~ dM'^T) + DW^T Q + (DA + DA^T) K,
//                                                                         DA = G^- o dA,  dA = -tril(dR V~^T, -1),
// the adjoints of the coefficient vectors as row sums (e.g. d abar_r = -sum_j dR X + scale sum_j dO (Q S), where
// sum_j dR_rj X_rj = sum_d K_rd (dR S^T)_rd reuses a product that dK needs anyway), the adjoints of the two masks
// d Geta = scale tril(dO V~^T) o (Q K^T), d G^- = dA o (K K^T), and from those the gate gradients (bwd_gates.cuh).
//
// Every product is M = 128 (a product costs the same for 64 rows): dO stacked on dR, Q stacked on K, V~_lo on V~_hi.
// Accumulator lane r belongs to row r of dQ, lane 64 + r to row r of dK.
//   Z_S = [dO; dR] S^T, Z_M = [dO; dR] M^T            state images read in place as MN-major operands
//   P = [dO; dR] V~^T, [Q K^T; K K^T]                 V~ as bf16 hi + lo
//   acc += [DW; DA] K                                 A from tensor memory (hi + lo), written over P by its readers
//   acc += [0; DW^T] Q + [0; DA^T] K                  the same matrices row-major in shared memory = MN-major A
//   V~ dS'^T, V~ dM'^T                                two passes each (hi, lo in lanes 64..127)
// Precision: q, k, dO, the states are bf16 as they stand; V~, DW, DA are hi + lo pairs; dR one bf16 value (as measured:
// its lo part changes no gradient's error).
//
// Shape of the kernel: what bounds it is the latency of a long serial list of short steps (load, product, epilogue),
// so TWO 256-thread CTAs share an SM (half the tensor memory, 110 KB of shared memory, 128 registers each) and fill each
// other's waits.  Three 32 KB areas are reused: A2 = Q, K (then the packed mask adjoints over Q); A1 = dO, dR, then the DW / DA
// tiles, dS', dM'; X = S, M, then V~.  Each next operand is fetched under the epilogue of the product before it.
#include <cstring>
#include <type_traits>

#include "bwd_gates.cuh"
#include "mdn_common.cuh"
#include "tc_utils.cuh"

namespace mdn {
namespace {

using namespace tc;
typedef __nv_bfloat16 bf16;

constexpr int kD = 128, kThreads = kGateThreads;
constexpr uint32_t kVecBytes = 24 * C * 4;
constexpr uint32_t kOffVec = 0, kOffDiag = kVecBytes, kOffA2 = 7168, kOffA1 = kOffA2 + 32768, kOffX = kOffA1 + 32768;
constexpr uint32_t kSmem = kOffX + 32768 + 1024;
static_assert(kOffDiag + C * 4 <= kOffA2 && kSmem <= 110 * 1024, "two CTAs per SM");
constexpr uint32_t kColAcc = 0, kColB = 128, kColP = 128, kColQK = 192, kCols = 256;
static_assert(kGateScratch * 4 <= 32768, "the gate stage's scratch lies in A1");

struct TcArgs {
  ChunkGeom g;
  const float* beta; const float* log_alpha; const float* log_mu; const float* eta;
  const float* coef;
  const uint8_t* fwd_states; const uint8_t* adj_states;   // state images per chunk slot
  int32_t* status;                                        // the forward workspace's status word
  float scale;
  void* dq; void* dk;
  int align;                                              // of dq, dk: 8, 16 or 32 bytes
  GateOut gates;
};

// 32 consecutive values of a row to global memory
template <typename TG> __device__ __forceinline__ void store_row32(TG* dst, const float2 (&x)[16], int align);
__device__ __forceinline__ void st_v8(void* p, const uint32_t (&w)[8], int align) {
  if (align == 32) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]),
                 "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
  } else if (align == 16) {
    static_cast<uint4*>(p)[0] = make_uint4(w[0], w[1], w[2], w[3]);
    static_cast<uint4*>(p)[1] = make_uint4(w[4], w[5], w[6], w[7]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) static_cast<uint2*>(p)[i] = make_uint2(w[2 * i], w[2 * i + 1]);
  }
}
template <> __device__ __forceinline__ void store_row32<bf16>(bf16* dst, const float2 (&x)[16], int align) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    uint32_t w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = pack_bf16(x[8 * i + e].x, x[8 * i + e].y);
    st_v8(dst + 16 * i, w, align);
  }
}
template <> __device__ __forceinline__ void store_row32<float>(float* dst, const float2 (&x)[16], int align) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint32_t w[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) { w[2 * e] = __float_as_uint(x[4 * i + e].x); w[2 * e + 1] = __float_as_uint(x[4 * i + e].y); }
    st_v8(dst + 8 * i, w, align);
  }
}

__device__ __forceinline__ float2 unpack2(uint32_t w) { return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }
__device__ __forceinline__ float2 f2(uint32_t a, uint32_t b) { return make_float2(__uint_as_float(a), __uint_as_float(b)); }

// index of element (r, i), i < r, of a packed strictly lower triangle.  Thirty-two consecutive rows of one column lie in
// thirty-two different banks (triangular numbers are a permutation modulo a power of two).
__device__ __forceinline__ int tri(int r, int i) { return ((r * (r - 1)) >> 1) + i; }

template <typename TG>
__global__ void __launch_bounds__(kThreads, 2) bwd_chunk_tc_kernel(const TcArgs a, const __grid_constant__ CUtensorMap map_q,
                                                                  const __grid_constant__ CUtensorMap map_k,
                                                                  const __grid_constant__ CUtensorMap map_do,
                                                                  const __grid_constant__ CUtensorMap map_dr,
                                                                  const __grid_constant__ CUtensorMap map_vt) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t bars[2];   // loads; products
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const int H = a.g.H, slot = blockIdx.x / H, h = blockIdx.x % H;
  grid_dependency_wait();
  const SlotInfo si = slot_info(a.g, slot);
  if (si.seq < 0) return;
  const int n = si.n;
  int slot0, nch;
  seq_chunks(a.g, si.seq, &slot0, &nch);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int L = (warp & 3) * 32 + lane, hf = warp >> 2;   // the thread's accumulator lane; its half of the columns
  const bool k_row = L >= 64;                             // a row of dK (else of dQ)
  const int r = L & 63;
  const bool live = r < n;
  const uint32_t sb = smem_u32(smem), bar_l = smem_u32(&bars[0]), bar_m = smem_u32(&bars[1]);
  float* vec = reinterpret_cast<float*>(smem + kOffVec);
  float* ge_diag = reinterpret_cast<float*>(smem + kOffDiag);
  float* gm_tri = reinterpret_cast<float*>(smem + kOffA2);            // packed d G^-, d Geta over the two halves of Q
  float* ge_tri = reinterpret_cast<float*>(smem + kOffA2 + 16384);
  auto V = [&](int which) { return vec + which * C; };
  auto tok = [&](int rr) { return (size_t)(si.tok0 + rr) * H + h; };
  const uint8_t* imgS = a.fwd_states + ((size_t)slot * H + h) * 65536;
  const int e_real = slot0 + (nch - 1 - si.local);   // this chunk in the adjoint chain's mirrored order
  const uint8_t* imgdM = a.adj_states + ((size_t)e_real * H + h) * 65536;   // roles exchanged in the adjoint run
  const uint8_t* imgdS = imgdM + 32768;
  const float scale = a.scale;

  auto load_image = [&](uint32_t off, const uint8_t* img) {   // one thread
    mbar_arrive_expect_tx(bar_l, 32768);
    bulk_load(sb + off, img, 16384, bar_l);
    bulk_load(sb + off + 16384, img + 16384, 16384, bar_l);
  };
  if (tid == 0) {
    abort_flag = 0;
    mbar_init(bar_l, 1);
    mbar_init(bar_m, 1);
    mbar_fence_init();
    mbar_arrive_expect_tx(bar_l, 3 * 32768);
    for (int j = 0; j < 2; ++j) {
      tma_load_2d(sb + kOffA1 + j * 16384, &map_do, h * kD + 64 * j, si.tok0, bar_l);
      tma_load_2d(sb + kOffA1 + j * 16384 + 8192, &map_dr, h * kD + 64 * j, si.tok0, bar_l);
      bulk_load(sb + kOffX + j * 16384, imgS + j * 16384, 16384, bar_l);
    }
    for (int j = 0; j < 2; ++j) {
      tma_load_2d(sb + kOffA2 + j * 16384, &map_q, h * kD + 64 * j, si.tok0, bar_l);
      tma_load_2d(sb + kOffA2 + j * 16384 + 8192, &map_k, h * kD + 64 * j, si.tok0, bar_l);
    }
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_slot), kCols);
    tc_fence_before_sync();
  }
  uint4 adj[8];   // the thread's 16-byte pieces of dS' (see dots below): under way with the tiles
#pragma unroll
  for (int i = 0; i < 8; ++i) adj[i] = __ldg(reinterpret_cast<const uint4*>(imgdS + (tid + kThreads * i) * 16));
  for (int i = tid; i < 24 * C; i += kThreads) vec[i] = 0.f;
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
  const uint32_t tl = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + hf * 64;   // the thread's lane, its 64 columns of a 128-wide result
  if (tid < C) {   // (all loads before the first store: they must not wait for one another)
    const float* cf = a.coef + ((size_t)slot * H + h) * MDN_NUM_COEF * C;
    const int t = tid;
    const bool in = t < n;
    const size_t gi = tok(in ? t : 0);
    const float x0 = __ldg(cf + kAbar * C + t), x1 = __ldg(cf + kB * C + t), x2 = __ldg(cf + kAlphaBPrev * C + t);
    const float x3 = __ldg(cf + kGS * C + t), x4 = __ldg(cf + kGM * C + t), x5 = __ldg(cf + kMubar * C + t);
    const float x6 = __ldg(cf + kB * C + max(t - 1, 0));
    const float ga = __ldg(a.log_alpha + gi), gm = __ldg(a.log_mu + gi), gb = __ldg(a.beta + gi), ge = a.eta ? __ldg(a.eta + gi) : 1.f;
    V(vAbar)[t] = x0; V(vB)[t] = x1; V(vP)[t] = x2;
    V(vGS)[t] = in ? x3 : 0.f; V(vGM)[t] = in ? x4 : 0.f; V(vMubar)[t] = x5;
    V(vAlpha)[t] = in ? expf(ga) : 1.f; V(vMu)[t] = in ? expf(gm) : 1.f;
    V(vBeta)[t] = in ? gb : 0.f; V(vEta)[t] = in ? ge : 0.f;
    V(vBprev)[t] = t > 0 ? x6 : 0.f;
  }

  uint32_t ph_l = 0, ph_m = 0;
  bool good = true;
  // All threads wait for the next load / product phase and learn whether everybody's wait succeeded (also a barrier).  The
  // lanes of a warp can leave the polling loop at different times, and a block barrier does not bring them together again: the
  // warp-collective tensor-memory loads that follow need the __syncwarp (without it they ran on parts of a warp, which
  // ended in an illegal memory access).
  auto wait_all = [&](uint32_t bar, uint32_t& ph) {
    const bool mine = mbar_wait(bar, ph, &abort_flag);
    __syncwarp();
    good = __syncthreads_and(mine) != 0;
    __syncwarp();
    ph ^= 1;
    tc_fence_after_sync();
    return good;
  };
  const uint32_t id_nn = idesc_bf16(128, 128, false, true, false), id_64 = idesc_bf16(128, 64, false, false, false);
  const uint32_t id_tn = idesc_bf16(128, 128, true, true, false);
  // Products are issued by one elected lane of warp 0 while the whole warp walks the same code: addresses made warp-uniform
  // here stay in uniform registers (a single thread's descriptor arithmetic took longer than its products)
  const uint32_t usb = __shfl_sync(0xffffffffu, sb, 0), utm = __shfl_sync(0xffffffffu, tmem, 0);
  const bool issuer = warp == 0;
  auto half = [&](uint32_t off, int k) { return smem_desc_sw128(usb + off + (k >> 2) * 16384, 16, 1024) + 2 * (k & 3); };   // K-major, 64-column halves

  // sum over the thread's share of <global image, shared image>
  auto dot8 = [&](const uint4& x, const uint4& y, float2& s) {
    s = __ffma2_rn(unpack2(x.x), unpack2(y.x), s); s = __ffma2_rn(unpack2(x.y), unpack2(y.y), s);
    s = __ffma2_rn(unpack2(x.z), unpack2(y.z), s); s = __ffma2_rn(unpack2(x.w), unpack2(y.w), s);
  };
  // the thread's 32-column pieces of an adjoint image, fetched long before the state they meet has arrived in X
  auto fetch8 = [&](const uint8_t* g, uint4 (&x)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = __ldg(reinterpret_cast<const uint4*>(g + (tid + kThreads * i) * 16));
  };
  auto dots = [&](const uint4 (&x)[8], float2& s) {
#pragma unroll
    for (int i = 0; i < 8; ++i) dot8(x[i], *reinterpret_cast<const uint4*>(smem + kOffX + (tid + kThreads * i) * 16), s);
  };
  auto add_dot = [&](float2 s, float* dst, float sign) {
    float x = s.x + s.y;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    if (lane == 0) atomicAdd(dst, sign * x);
  };
  // 32 columns (32 c .. of the thread's 64) of its row of [Q; K], as float pairs
  auto qk_row = [&](int c, float2 (&x)[16]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint4 w = *reinterpret_cast<const uint4*>(smem + kOffA2 + hf * 16384 + L * 128 + (((4 * c + u) ^ (L & 7)) << 4));
      x[4 * u] = unpack2(w.x); x[4 * u + 1] = unpack2(w.y); x[4 * u + 2] = unpack2(w.z); x[4 * u + 3] = unpack2(w.w);
    }
  };
  // One product's epilogue: z = 64 columns at col; acc (at kColAcc) = w z (first) or acc + w z; a row sum of z o [Q; K] goes
  // to dvec.  out: the finished row leaves for global memory instead of returning to tensor memory.
  auto epilogue = [&](uint32_t col, bool first, float w, float* dvec, float sign, TG* out) {
    float2 s = make_float2(0.f, 0.f);
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      uint32_t z[32];
      tmem_ld32(tl + col + 32 * c, z);
      float2 x[16];
      qk_row(c, x);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 16; ++i) s = __ffma2_rn(f2(z[2 * i], z[2 * i + 1]), x[i], s);
      if (first) {
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = __fmul2_rn(make_float2(w, w), f2(z[2 * i], z[2 * i + 1]));
      } else {
        uint32_t acc[32];
        tmem_ld32(tl + kColAcc + 32 * c, acc);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = __ffma2_rn(make_float2(w, w), f2(z[2 * i], z[2 * i + 1]), f2(acc[2 * i], acc[2 * i + 1]));
      }
      if (out != nullptr) {
        if (live) store_row32<TG>(out + 32 * c, x, a.align);
        __syncwarp();
      } else {
        uint32_t y[32];
#pragma unroll
        for (int i = 0; i < 16; ++i) { y[2 * i] = __float_as_uint(x[i].x); y[2 * i + 1] = __float_as_uint(x[i].y); }
        tmem_st32(tl + kColAcc + 32 * c, y);
      }
    }
    if (out == nullptr) tmem_wait_st();
    tc_fence_before_sync();
    if (live) atomicAdd(dvec + r, sign * (s.x + s.y));
  };

  do {
    // ---- Z_S
    if (!wait_all(bar_l, ph_l)) break;
    if (issuer && elect_one()) {
      const uint64_t dB = smem_desc_sw128(usb + kOffX, 16384, 1024);
#pragma unroll
      for (int k = 0; k < 8; ++k) umma_ss(utm + kColAcc, half(kOffA1, k), dB + 128 * k, id_nn, k > 0);
      umma_commit(bar_m);
    }
    float2 s0 = make_float2(0.f, 0.f), s1 = s0, s2 = s0;
    dots(adj, s1);                                                 // <dS', S>
    if (!wait_all(bar_m, ph_m)) break;   // (also: every thread is done with S)
    if (tid == 0) { fence_proxy_async_smem(); load_image(kOffX, imgS + 32768); }
    add_dot(s1, V(vdAbar) + n - 1, 1.f);
    epilogue(kColAcc, true, k_row ? -V(vAbar)[r] : scale * V(vAbar)[r], V(vdAbar), k_row ? -1.f : scale, nullptr);

    // ---- Z_M
    uint4 adj2[8];
    fetch8(imgdS, adj);
    fetch8(imgdM, adj2);
    if (!wait_all(bar_l, ph_l)) break;
    if (issuer && elect_one()) {
      const uint64_t dB = smem_desc_sw128(usb + kOffX, 16384, 1024);
#pragma unroll
      for (int k = 0; k < 8; ++k) umma_ss(utm + kColB, half(kOffA1, k), dB + 128 * k, id_nn, k > 0);
      umma_commit(bar_m);
    }
    dots(adj2, s0);                                                // <dM', M>
    dots(adj, s2);                                                 // <dS', M>
    if (!wait_all(bar_m, ph_m)) break;
    if (tid == 0) {
      fence_proxy_async_smem();
      mbar_arrive_expect_tx(bar_l, 32768);
      tma_load_2d(sb + kOffX, &map_vt, h * kD, slot * C, bar_l);   // V~, fp32
    }
    add_dot(s0, V(vdMubar) + n - 1, 1.f);
    add_dot(s2, V(vdB) + n - 1, -1.f);
    epilogue(kColB, false, k_row ? V(vP)[r] : -scale * V(vB)[r], V(k_row ? vdP : vdB), k_row ? 1.f : -scale, nullptr);

    // ---- the thread's 32 columns (32 hf ..) of its row of scale Gamma eta (dQ rows) or G^- (dK rows), right to left:
    // gamma_{rp,i} = mu_{i+1} gamma_{rp,i+1} + beta_i prod_{i<l<=rp} alpha_l
    float f[32];
    {
      const int rp = live ? (k_row ? r - 1 : r) : -1;
      const float seed = k_row ? V(vAlpha)[r] : scale;
      float G = 0.f, al = 0.f, mu_next = 0.f;
      auto walk = [&](int from, auto keep_tag) {   // 32 columns from + 31 down to from
        constexpr bool kKeep = decltype(keep_tag)::value;
#pragma unroll
        for (int i4 = 28; i4 >= 0; i4 -= 4) {
          const float4 a4 = *reinterpret_cast<const float4*>(V(vAlpha) + from + i4), b4 = *reinterpret_cast<const float4*>(V(vBeta) + from + i4);
          const float4 m4 = *reinterpret_cast<const float4*>(V(vMu) + from + i4), e4 = *reinterpret_cast<const float4*>(V(vEta) + from + i4);
          const float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w}, mv[4] = {m4.x, m4.y, m4.z, m4.w},
                      ev[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
          for (int e = 3; e >= 0; --e) {
            al = (from + i4 + e == rp) ? seed : al;   // (stays 0 until the walk reaches the row's last column)
            G = fmaf(mu_next, G, bv[e] * al);
            al *= av[e];
            if constexpr (kKeep) f[i4 + e] = G * ev[e];
            mu_next = mv[e];
          }
        }
      };
      const bool upper = (warp & 1) != 0;   // rows 32..63; the others end at column 31
      if (hf == 1) {
        if (upper) walk(32, std::true_type{});
        else {
#pragma unroll
          for (int i = 0; i < 32; ++i) f[i] = 0.f;
        }
      } else {
        if (upper) walk(32, std::false_type{});
        walk(0, std::true_type{});
      }
    }
    // ---- V~: fp32 -> bf16 hi, lo tiles in place (rows past the chunk's end cleared); half j: lo at 16384 j, hi 8192 behind it
    if (!wait_all(bar_l, ph_l)) break;
    {
      float4 x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = *reinterpret_cast<const float4*>(smem + kOffX + (tid + kThreads * i) * 16);
      __syncthreads();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int idx = tid + kThreads * i, rr = idx >> 5, c = (idx & 31) * 4;
        uint2 ph = make_uint2(0u, 0u), pl = ph;
        if (rr < n) {
          split_pack_bf16(make_float2(x[i].x, x[i].y), ph.x, pl.x);
          split_pack_bf16(make_float2(x[i].z, x[i].w), ph.y, pl.y);
        }
        uint8_t* dst = smem + kOffX + (c >> 6) * 16384 + sw128_offset(rr, c & 63);
        *reinterpret_cast<uint2*>(dst) = pl;
        *reinterpret_cast<uint2*>(dst + 8192) = ph;
      }
    }
    fence_proxy_async_smem();
    tc_fence_before_sync();   // (the epilogue's tensor-memory reads of kColB)
    __syncthreads();
    // ---- P = [dO; dR] V~^T, [Q K^T; K K^T]
    if (issuer && elect_one()) {
      tc_fence_after_sync();
#pragma unroll
      for (int k = 0; k < 8; ++k) umma_ss(utm + kColP, half(kOffA1, k), half(kOffX + 8192, k), id_64, k > 0);
#pragma unroll
      for (int k = 0; k < 8; ++k) umma_ss(utm + kColP, half(kOffA1, k), half(kOffX, k), id_64, true);
#pragma unroll
      for (int k = 0; k < 8; ++k) umma_ss(utm + kColQK, half(kOffA2, k), half(kOffA2 + 8192, k), id_64, k > 0);
      umma_commit(bar_m);
    }
    if (!wait_all(bar_m, ph_m)) break;
    // ---- DW, DA: hi + lo over P in tensor memory (row operand), and row-major in shared memory (transposed operand): a zero
    // block, DW hi, DW lo, DA hi of 8 KB each in A1.  f becomes the row of d Geta / d G^-.
    {
      const uint32_t tp = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + 32 * hf;
      uint32_t hi[16], lo[16];
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t p[16], x[16];
        tmem_ld16(tp + kColP + 16 * c, p);
        tmem_ld16(tp + kColQK + 16 * c, x);
        tmem_wait_ld();
        const int last = live ? (k_row ? r - 1 : r) - 32 * hf - 16 * c : -1;   // the mask's last column, relative to these sixteen
        const float sg = k_row ? -1.f : 1.f, sm = k_row ? -1.f : scale;
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
          float d[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float pv = i + e <= last ? __uint_as_float(p[i + e]) : 0.f;
            d[e] = sg * f[16 * c + i + e] * pv;
            f[16 * c + i + e] = i + e <= last ? sm * pv * __uint_as_float(x[i + e]) : 0.f;
          }
          split_pack_bf16(make_float2(d[0], d[1]), hi[8 * c + i / 2], lo[8 * c + i / 2]);
        }
      }
      __syncwarp();
      tmem_st16(tp + kColP, hi);
      tmem_st16(tp + kColP + 16, lo);
      uint8_t* zero = smem + kOffA1;
      uint8_t* dst = zero + (k_row ? 3 * 8192 : 8192) + r * 128;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t off = ((4 * hf + u) ^ (r & 7)) << 4;
        *reinterpret_cast<uint4*>(dst + off) = make_uint4(hi[4 * u], hi[4 * u + 1], hi[4 * u + 2], hi[4 * u + 3]);
        if (!k_row) *reinterpret_cast<uint4*>(dst + 8192 + off) = make_uint4(lo[4 * u], lo[4 * u + 1], lo[4 * u + 2], lo[4 * u + 3]);
        else *reinterpret_cast<uint4*>(zero + r * 128 + off) = make_uint4(0u, 0u, 0u, 0u);
      }
      tmem_wait_st();
    }
    fence_proxy_async_smem();
    tc_fence_before_sync();
    __syncthreads();
    // ---- acc += [DW; DA] K + [0; DW^T] Q + [0; DA^T] K
    if (issuer && elect_one()) {
      tc_fence_after_sync();
      const uint64_t dK = smem_desc_sw128(usb + kOffA2 + 8192, 16384, 1024), dQ = smem_desc_sw128(usb + kOffA2, 16384, 1024);
#pragma unroll
      for (int part = 0; part < 2; ++part)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          umma_ts(utm + kColAcc, utm + kColP + 32 * (k >> 1) + 16 * part + 8 * (k & 1), dK + 128 * k, id_nn, true);
#pragma unroll
      for (int m = 1; m < 4; ++m) {   // the zero block is rows 0..63 of A, m blocks further on lie rows 64..127
        const uint64_t dA = smem_desc_sw128(usb + kOffA1, m * 8192, 1024);
#pragma unroll
        for (int k = 0; k < 4; ++k) umma_ss(utm + kColAcc, dA + 128 * k, (m == 3 ? dK : dQ) + 128 * k, id_tn, true);
      }
      umma_commit(bar_m);
    }
    if (!wait_all(bar_m, ph_m)) break;
    if (tid == 0) { fence_proxy_async_smem(); load_image(kOffA1, imgdS); }
    // Q is dead: the mask adjoints take its place, packed
    if (!k_row && (r >> 5) == hf) {   // the diagonal element is in the half that holds column r
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (i == (r & 31)) ge_diag[r] = f[i];
    }
    {
      float* dst = (k_row ? gm_tri : ge_tri) + tri(r, 32 * hf);
      const int lim = r - 32 * hf;
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (i < lim) dst[i] = f[i];
    }
    __syncwarp();
    if (!k_row) {   // dQ is finished
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t acc[32];
        tmem_ld32(tl + kColAcc + 32 * c, acc);
        tmem_wait_ld();
        float2 x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = f2(acc[2 * i], acc[2 * i + 1]);
        if (live) store_row32<TG>(static_cast<TG*>(a.dq) + tok(r) * kD + 64 * hf + 32 * c, x, a.align);
        __syncwarp();
      }
    }
    // ---- V~ dS'^T, V~ dM'^T (lanes 64..127: hi from [lo; hi], then lo from the tile that starts 8 KB earlier)
    bool broke = false;
#pragma unroll 1
    for (int which = 0; which < 2; ++which) {
      if (!wait_all(bar_l, ph_l)) { broke = true; break; }
      if (issuer && elect_one()) {
        const uint64_t dB = smem_desc_sw128(usb + kOffA1, 16384, 1024);
#pragma unroll
        for (int k = 0; k < 8; ++k) umma_ss(utm + kColB, half(kOffX, k), dB + 128 * k, id_nn, k > 0);
#pragma unroll
        for (int k = 0; k < 8; ++k) umma_ss(utm + kColB, half(kOffX - 8192, k), dB + 128 * k, id_nn, true);
        umma_commit(bar_m);
      }
      if (!wait_all(bar_m, ph_m)) { broke = true; break; }
      if (which == 0 && tid == 0) { fence_proxy_async_smem(); load_image(kOffA1, imgdM); }
      if (k_row)
        epilogue(kColB, false, which ? -V(vGM)[r] : V(vGS)[r], V(which ? vdGM : vdGS), which ? -1.f : 1.f,
                 which ? static_cast<TG*>(a.dk) + tok(r) * kD + 64 * hf : nullptr);
    }
    if (broke) break;
  } while (false);

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after_sync();
    tmem_dealloc(tmem, kCols);
  }
  if (!good) {
    if (tid == 0) atomicCAS(a.status, kDevOk, kDevTimeout);
    return;
  }
  gate_gradients(vec, [&](int rr, int i) { return ge_tri[rr > i ? tri(rr, i) : 0]; }, [&](int i) { return ge_diag[i]; },
                 [&](int rr, int i) { return gm_tri[rr > i ? tri(rr, i) : 0]; }, reinterpret_cast<float*>(smem + kOffA1), n, tok(0), H, a.gates);
}

}  // namespace

cudaError_t launch_bwd_chunk_tc(const Plan& fwd, const void* q, const void* k, const void* d_o, const float* beta,
                                const float* log_alpha, const float* log_mu, const float* eta, const void* fwd_states,
                                const float* fwd_vt, const void* adj_states, const void* dr_bf16, void* dq, void* dk, bool grads_bf16,
                                float* dbeta, float* dlog_alpha, float* dlog_mu, float* deta, int* launches) {
  const uint64_t tokens = (uint64_t)fwd.p.B * fwd.p.T, row = (uint64_t)fwd.p.H * kD;
  CUtensorMap mq, mk, mdo, mdr, mvt;
  if (!encode_tma_2d_bf16(&mq, TmaMap2D{q, row, tokens, row * 2, 64, 64, true}) ||
      !encode_tma_2d_bf16(&mk, TmaMap2D{k, row, tokens, row * 2, 64, 64, true}) ||
      !encode_tma_2d_bf16(&mdo, TmaMap2D{d_o, row, tokens, row * 2, 64, 64, true}) ||
      !encode_tma_2d_bf16(&mdr, TmaMap2D{dr_bf16, row, tokens, row * 2, 64, 64, true}) ||
      !encode_tma_2d(&mvt, TmaMap2D{fwd_vt, row, (uint64_t)fwd.geom.num_slots * C, row * 4, 128, 64, false}, true))
    return cudaErrorInvalidValue;
  TcArgs a;
  a.g = fwd.geom;
  a.beta = beta; a.log_alpha = log_alpha; a.log_mu = log_mu; a.eta = eta;
  a.coef = reinterpret_cast<const float*>(fwd.ws + fwd.lay.off_coef);
  a.fwd_states = static_cast<const uint8_t*>(fwd_states);
  a.adj_states = static_cast<const uint8_t*>(adj_states);
  a.status = reinterpret_cast<int32_t*>(fwd.ws + fwd.lay.off_status);
  a.scale = fwd.p.scale;
  a.dq = dq; a.dk = dk;
  const uintptr_t at = reinterpret_cast<uintptr_t>(dq) | reinterpret_cast<uintptr_t>(dk);
  if (at & 7) return cudaErrorInvalidValue;
  a.align = at & 15 ? 8 : at & 31 ? 16 : 32;
  a.gates = GateOut{dbeta, dlog_alpha, dlog_mu, deta};
  auto launch = [&](auto kern) -> cudaError_t {
    cudaError_t e = allow_smem<(int)kSmem>(kern);
    if (e != cudaSuccess) return e;
    e = launch_pdl(kern, dim3((unsigned)fwd.geom.num_slots * fwd.p.H), dim3(kThreads), kSmem, fwd.stream, a, mq, mk, mdo, mdr, mvt);
    if (e == cudaSuccess) ++*launches;
    return e;
  };
  return grads_bf16 ? launch(bwd_chunk_tc_kernel<bf16>) : launch(bwd_chunk_tc_kernel<float>);
}

}  // namespace mdn
