// Exact backward (mdn_chunk_bwd): every gradient in fp32, chunk by chunk, any i/o type and dk, dv in {64, 128}.
//
// The chunk form of Section 3.1 differentiated matrix by matrix.  With dS', dM' the adjoints at a chunk's end,
//     dV~ = W^T dO + g_S.(K dS') - g_M.(K dM'),   dR = T^T dV~ = dV,
//     dS  = abar_C dS' - K^T (abar.dR) + scale Q^T (abar.dO),
//     dM  = -b_C dS' + mubar_C dM' + K^T (p.dR) - scale Q^T (b.dO),
//     dQ  = scale (abar.(dO S^T) - b.(dO M^T)) + DW K,                    DW = scale Geta o tril(dO V~^T),
//     dK  = -abar.(dR S^T) + p.(dR M^T) + g_S.(V~ dS'^T) - g_M.(V~ dM'^T) + DW^T Q + (DA + DA^T) K,
//                                                                         DA = G^- o dA,  dA = -tril(dR V~^T, -1),
// the coefficient vectors' adjoints as row sums of products that dQ, dK need anyway, and the gate gradients from those
// by the scans of Eq. 10 in reverse (bwd_gates.cuh).  Five kernels:
//   status / chunk map;  intra_simt (scan, T, T^T, W^T);  chain_simt without output terms (the states at every chunk's start, V~);
//   the adjoint chain (dS', dM' at every chunk's end, dR);  the per-chunk kernel (everything else, all chunks in parallel).
//
// Why: the serial part of a backward is two walks over the chunks.  The token-by-token form this replaces was serial
// over tokens (3.4 us per token and chain whatever the GPU's size: 3.4 ms for T = 1023, B H = 16); here 64 tokens cost
// one chunk step of either chain, and the bulk of the arithmetic (20 of 28 products) is parallel over chunks.
#include "bwd_gates.cuh"
#include "simt_tile.cuh"

namespace mdn {
namespace {

// ================================================================================================ adjoint chain
struct AdjArgs {
  ChunkGeom g;
  const void* q; const void* k; const void* d_o;
  bool in_bf16, do_bf16;
  int dv;
  const float* coef; const float* TT; const float* WT;
  const float* dSf; const float* dMf;
  float scale;
  float* adj;            // [slot][H][2][dk][dv]: dS', dM' at the chunk's end
  float* dv_out;         // dR = dL/dv, [B,T,H,dv]
  float* dS0; float* dM0;
};

template <int DK, int NV> struct AdjSmem {   // float offsets; the K tile is twice buffered for fp32 input, for bf16 the raw
  static constexpr int LDK = DK + 4;         // staging area is the second buffer
  static constexpr int Q = 0, TT = Q + C * LDK, WT = TT + C * kLT, D = WT + C * kLT, Dot = D + 2 * NV * LDK, Zt = Dot + NV * kLT,
                       Wd = Zt + NV * kLT, cv = Wd + 2 * C * NV * 4, K = cv + 2 * kChainCoefs * C;
  static constexpr size_t bytes(bool bf16) {
    return (size_t)(K + (bf16 ? 1 : 2) * C * LDK) * 4 + (bf16 ? (size_t)2 * C * DK * 2 : 0);
  }
};

// One CTA per (sequence, head, NV value columns), chunks from last to first; the columns of dS', dM' stay in shared
// memory.  Same structure and products as the forward chain (chain_simt.cu); the two Q terms make its state update
// twice as long (rows of K, then rows of Q).
template <int DK, int NV>
__global__ void __launch_bounds__(kSimtThreads, DK == 64 ? 2 : 1) adj_chain_kernel(const AdjArgs a) {
  extern __shared__ __align__(16) float sm[];
  using L = AdjSmem<DK, NV>;
  constexpr int LDK = L::LDK, JT = NV / 8;
  constexpr int DT = (DK == 64 && NV == 8) ? 2 : 4, JC = NV * DK / (kSimtThreads * DT), JG = NV / JC;
  float* Qs = sm + L::Q;
  float* TTm = sm + L::TT;
  float* WTm = sm + L::WT;
  float* Ds = sm + L::D;       // [2 NV (columns of dS', then of dM')][LDK]
  float* Dot = sm + L::Dot;    // dO^T
  float* Zt = sm + L::Zt;      // dV~^T
  float4* Wd = reinterpret_cast<float4*>(sm + L::Wd);   // [128 rows (K, then Q)][NV]: weights of the update of dS', dM', each twice
  uint8_t* raw = reinterpret_cast<uint8_t*>(sm + L::K + C * LDK);
  uint8_t* rawQ = raw + C * DK * 2;

  const int tid = threadIdx.x, jg = tid & 7, rs = tid >> 3;
  const int H = a.g.H, DV = a.dv, NVB = DV / NV;
  const int vb = blockIdx.x % NVB, h = (blockIdx.x / NVB) % H, seq = blockIdx.x / (NVB * H);
  const int j0 = vb * NV;
  grid_launch_dependents();
  grid_dependency_wait();
  const SeqInfo sq = seq_info(a.g, seq);
  const size_t st_off = ((size_t)seq * H + h) * DK * DV;
  const size_t es = a.in_bf16 ? 2 : 4;
  const int nch = sq.nchunks;
  auto src_of = [&](const void* p, int c) {
    return static_cast<const void*>(static_cast<const uint8_t*>(p) + ((size_t)(sq.tok0 + c * C) * H + h) * DK * es);
  };
  auto k_tile = [&](int c) { return sm + L::K + (a.in_bf16 ? 0 : (c & 1) * C * LDK); };
  auto fetch_k = [&](int c) {
    load_rows<DK>(k_tile(c), raw, src_of(a.k, c), a.in_bf16, (size_t)H * DK, min(C, sq.len - c * C), tid);
    const float* cf = a.coef + ((size_t)(sq.slot0 + c) * H + h) * MDN_NUM_COEF * C;
    if (tid < kChainCoefs * C / 4) cp16(sm + L::cv + (c & 1) * kChainCoefs * C + tid * 4, cf + tid * 4, true);
  };
  auto mat = [&](int c) { return ((size_t)(sq.slot0 + c) * H + h) * C * C; };
  float dnext[2][JT];
  auto load_do = [&](int c) {   // this thread's elements of the chunk's dO: rows rs + 32 i, columns jg + 8 jj
    const int n = min(C, sq.len - c * C);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int jj = 0; jj < JT; ++jj) {
        const int r = rs + 32 * i;
        dnext[i][jj] = r < n ? load_io(a.d_o, ((size_t)(sq.tok0 + c * C + r) * H + h) * DV + j0 + jg + 8 * jj, a.do_bf16) : 0.f;
      }
  };

  if (nch > 0) {
    fetch_k(nch - 1);
    load_mat(WTm, a.WT + mat(nch - 1), tid);
    load_mat(TTm, a.TT + mat(nch - 1), tid);
    cp_commit();
    load_do(nch - 1);
  }
  for (int i = tid; i < 2 * NV * DK; i += kSimtThreads) {
    const int jj = i % NV, d = (i / NV) % DK, which = i / (NV * DK);
    const float* src = which ? a.dMf : a.dSf;
    Ds[(which * NV + jj) * LDK + d] = src ? src[st_off + (size_t)d * DV + j0 + jj] : 0.f;
  }

  for (int c = nch - 1; c >= 0; --c) {
    const int n = min(C, sq.len - c * C);
    const size_t slot_h = (size_t)(sq.slot0 + c) * H + h;
    float* Ks = k_tile(c);
    const float* cv = sm + L::cv + (c & 1) * kChainCoefs * C;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int jj = 0; jj < JT; ++jj) Dot[(jg + 8 * jj) * kLT + rs + 32 * i] = dnext[i][jj];
    cp_wait<0>();
    __syncthreads();   // tiles landed; the previous step's readers are done, its adjoints are written
    if (a.in_bf16) {
      widen_tile<DK>(Ks, raw, tid);
      __syncthreads();
    }
    if (c > 0) fetch_k(c - 1);
    load_rows<DK>(Qs, rawQ, src_of(a.q, c), a.in_bf16, (size_t)H * DK, n, tid);
    cp_commit();
    {   // the adjoint pair at the chunk's end, [d][j]
      float* dst = a.adj + slot_h * 2 * DK * DV + j0;
      for (int i = tid; i < 2 * NV * DK; i += kSimtThreads) {
        const int j = i % NV, d = (i / NV) % DK, which = i / (NV * DK);
        dst[(size_t)which * DK * DV + (size_t)d * DV + j] = Ds[(which * NV + j) * LDK + d];
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {   // weights of the Q rows
      const int r = rs + 32 * i;
      const float ws = a.scale * cv[kAbar * C + r], wm = -a.scale * cv[kB * C + r];
#pragma unroll
      for (int jj = 0; jj < JT; ++jj) {
        const float x = dnext[i][jj];
        Wd[(C + r) * NV + jg + 8 * jj] = make_float4(ws * x, ws * x, wm * x, wm * x);
      }
    }

    // ---- 1: dV~ = W^T dO + g_S.(K dS') - g_M.(K dM'), rows rs + 32 i   (W^T is upper triangular)
    {
      float2 acc[2][2 * JT], wv[2][JT];
      zero2(acc); zero2(wv);
      dot_tile<2, 2 * JT>(acc, Ks + rs * LDK, 32 * LDK, Ds + jg * LDK, 8 * LDK, 0, DK / 4);
      dot_tile<2, JT>(wv, WTm + rs * kLT, 32 * kLT, Dot + jg * kLT, 8 * kLT, 8, 16);
      float2 lo[1][JT];
#pragma unroll
      for (int jj = 0; jj < JT; ++jj) lo[0][jj] = wv[0][jj];
      dot_tile<1, JT>(lo, WTm + rs * kLT, 0, Dot + jg * kLT, 8 * kLT, 0, 8);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = rs + 32 * i;
        const float gs = cv[kGS * C + r], gm = cv[kGM * C + r];
#pragma unroll
        for (int jj = 0; jj < JT; ++jj)
          Zt[(jg + 8 * jj) * kLT + r] = (i ? hsum(wv[1][jj]) : hsum(lo[0][jj])) + gs * hsum(acc[i][jj]) - gm * hsum(acc[i][JT + jj]);
      }
    }
    __syncthreads();
    if (c > 0) load_mat(WTm, a.WT + mat(c - 1), tid);   // W^T has been read
    cp_commit();

    // ---- 2: dR = T^T dV~  (upper triangular)
    {
      float2 acc[2][JT];
      zero2(acc);
      dot_tile<2, JT>(acc, TTm + rs * kLT, 32 * kLT, Zt + jg * kLT, 8 * kLT, 8, 16);
      float2 lo[1][JT];
#pragma unroll
      for (int jj = 0; jj < JT; ++jj) lo[0][jj] = acc[0][jj];
      dot_tile<1, JT>(lo, TTm + rs * kLT, 0, Zt + jg * kLT, 8 * kLT, 0, 8);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = rs + 32 * i;
        const float ws = -cv[kAbar * C + r], wm = cv[kAlphaBPrev * C + r];
#pragma unroll
        for (int jj = 0; jj < JT; ++jj) {
          const float x = i ? hsum(acc[1][jj]) : hsum(lo[0][jj]);
          const int j = jg + 8 * jj;
          if (r < n) a.dv_out[((size_t)(sq.tok0 + c * C + r) * H + h) * DV + j0 + j] = x;
          Wd[r * NV + j] = make_float4(ws * x, ws * x, wm * x, wm * x);
        }
      }
    }
    cp_wait<1>();   // K of the next step and Q are in
    __syncthreads();
    if (a.in_bf16) {
      widen_tile<DK>(Qs, rawQ, tid);
      __syncthreads();
    }
    if (c > 0) {
      load_mat(TTm, a.TT + mat(c - 1), tid);   // T^T has been read
      load_do(c - 1);
    }
    cp_commit();

    // ---- 3: the adjoint pair at the chunk's start, DT key rows x JC columns of both per thread (one owner per entry)
    {
      const int lane = tid & 31, warp = tid >> 5;
      constexpr int DB = DK / DT / 8;
      const int d0 = ((warp % DB) * 8 + (lane & 7)) * DT, jq = (warp / DB) * 4 + (lane >> 3);
      float2 acc[2 * JC][DT / 2];
      zero2(acc);
      auto update = [&](const float* kp, const float4* wp) {
#pragma unroll 4
        for (int r = 0; r < n; ++r) {
          float2 kv[DT / 2];
          if constexpr (DT == 4) {
            const float4 k4 = lds4(kp + r * LDK);
            kv[0] = make_float2(k4.x, k4.y); kv[1] = make_float2(k4.z, k4.w);
          } else {
            kv[0] = *reinterpret_cast<const float2*>(kp + r * LDK);
          }
#pragma unroll
          for (int jc = 0; jc < JC; ++jc) {
            const float4 w = wp[r * NV + JG * jc];
#pragma unroll
            for (int p = 0; p < DT / 2; ++p) {
              acc[2 * jc][p] = __ffma2_rn(kv[p], make_float2(w.x, w.y), acc[2 * jc][p]);
              acc[2 * jc + 1][p] = __ffma2_rn(kv[p], make_float2(w.z, w.w), acc[2 * jc + 1][p]);
            }
          }
        }
      };
      update(Ks + d0, Wd + jq);
      update(Qs + d0, Wd + C * NV + jq);
      const float aC = cv[kAbar * C + C - 1], bC = cv[kB * C + C - 1], mC = cv[kMubar * C + C - 1];
#pragma unroll
      for (int jc = 0; jc < JC; ++jc) {
        float* sp = Ds + (jq + JG * jc) * LDK + d0;
        float* mp = sp + NV * LDK;
#pragma unroll
        for (int p = 0; p < DT / 2; ++p) {
          const float2 s = *reinterpret_cast<float2*>(sp + 2 * p), m = *reinterpret_cast<float2*>(mp + 2 * p);
          const float2 ds = acc[2 * jc][p], dm = acc[2 * jc + 1][p];
          *reinterpret_cast<float2*>(sp + 2 * p) = make_float2(aC * s.x + ds.x, aC * s.y + ds.y);
          *reinterpret_cast<float2*>(mp + 2 * p) = make_float2(mC * m.x - bC * s.x + dm.x, mC * m.y - bC * s.y + dm.y);
        }
      }
    }
  }
  cp_wait<0>();
  __syncthreads();
  for (int i = tid; i < 2 * NV * DK; i += kSimtThreads) {
    const int jj = i % NV, d = (i / NV) % DK, which = i / (NV * DK);
    float* dst = which ? a.dM0 : a.dS0;
    if (dst) dst[st_off + (size_t)d * DV + j0 + jj] = Ds[(which * NV + jj) * LDK + d];
  }
}

// ============================================================================================== per-chunk kernel
struct ParArgs {
  ChunkGeom g;
  const void* q; const void* k; const void* d_o;
  bool in_bf16, do_bf16;
  const float* coef;
  const float* states; const float* adj;   // [slot][H][2][dk][dv]: S, M at the start; dS', dM' at the end
  const float* vt; const float* dr;        // V~ [slot][H][64][dv]; dR [B,T,H,dv]
  float scale;
  float* dq; float* dk;
  GateOut gates;
};

template <int DK, int DV> struct ParSmem {   // float offsets
  static constexpr int LDK = DK + 4, LDV = DV + 4, LB = 36, kMat = C * kLT;
  static constexpr int kStages = 3, kStage = DK * LB, kStageArea = kStages * kStage > 2 * kMat ? kStages * kStage : 2 * kMat;
  static constexpr int K = 0, Q = K + C * LDK, vec = Q + C * LDK, st = vec + 24 * C, tiles = st + kStageArea,
                       kTiles = 3 * C * LDV > 5 * kMat ? 3 * C * LDV : 5 * kMat, kFloats = tiles + kTiles;
  static_assert(kFloats * 4 <= 232448, "shared memory");
};

// One 256-thread CTA per (chunk, head).  The six products against states ([64 x dv] times [dv x dk]) stream the states
// through a three-stage ring of 32-column pieces; dO, dR, V~, K, Q stay in shared memory, dQ and dK in registers (4 rows x dk / 16
// columns per thread: 12 operand loads feed 64 packed FMAs per four terms).  Bound by the fp32 pipes: 9.5 M
// multiply-adds per chunk and head at dk = dv = 128.
template <int DK, int DV>
__global__ void __launch_bounds__(kSimtThreads, 1) bwd_exact_par_kernel(const ParArgs a) {
  extern __shared__ __align__(16) float sm[];
  using L = ParSmem<DK, DV>;
  constexpr int LDK = L::LDK, LDV = L::LDV, LB = L::LB, E2 = DK / 32, NP = DV / 32;
  float* Ks = sm + L::K;
  float* Qs = sm + L::Q;
  float* vec = sm + L::vec;
  float* Do = sm + L::tiles;
  float* Dr = Do + C * LDV;
  float* Vt = Dr + C * LDV;
  // after the streams / the products: 64 x 64 matrices
  float* Gam = sm + L::st;
  float* Mm = Gam + L::kMat;
  float* DW = sm + L::tiles;
  float* DWT = DW + L::kMat;
  float* DAS = DWT + L::kMat;   // DA + DA^T
  float* dGe = DAS + L::kMat;
  float* dGm = dGe + L::kMat;
  auto V = [&](int which) { return vec + which * C; };

  const int H = a.g.H, slot = blockIdx.x / H, h = blockIdx.x % H;
  grid_launch_dependents();
  grid_dependency_wait();
  const SlotInfo si = slot_info(a.g, slot);
  if (si.seq < 0) return;
  const int n = si.n;
  const int tid = threadIdx.x, lane = tid & 31;
  const int dg = (tid & 7) | (((tid >> 5) & 1) << 3), rl = ((tid >> 3) & 3) + 4 * (tid >> 6);   // columns dg.., rows rl + 16 i
  const size_t slot_h = (size_t)slot * H + h, tok_h = (size_t)si.tok0 * H + h;
  const float* fS = a.states + slot_h * 2 * DK * DV;
  const float* aS = a.adj + slot_h * 2 * DK * DV;
  const float scale = a.scale;

  // ---- the ring: piece p = (pass, 32 value columns); key row d of a state lies at ring row (d & 1) dk / 2 + d / 2, so that a
  // thread's column PAIRS (2 dg + 32 e, + 1) are rows dg + 16 e of either half: conflict-free loads, 8-byte stores
  auto fetch = [&](int p) {
    if (p < 6 * NP) {
      const int pass = p / NP, jb = p % NP;
      const float* src = (pass < 4 ? fS + (size_t)(pass & 1) * DK * DV : aS + (size_t)(pass & 1) * DK * DV) + jb * 32;
      float* dst = sm + L::st + (p % L::kStages) * L::kStage;
#pragma unroll
      for (int i = 0; i < DK * 8 / kSimtThreads; ++i) {
        const int idx = tid + i * kSimtThreads, d = idx >> 3, c4 = (idx & 7) * 4;
        cp16(dst + ((d & 1) * (DK / 2) + (d >> 1)) * LB + c4, src + (size_t)d * DV + c4, true);
      }
    }
    cp_commit();
  };
  auto load_io_rows = [&](auto width, float* tile, const void* src, bool bf16) {   // 64 rows of one head of an i/o tensor
    constexpr int D = decltype(width)::value;
    if (!bf16) { load_rows<D>(tile, nullptr, static_cast<const float*>(src) + tok_h * D, false, (size_t)H * D, n, tid); return; }
    for (int i = tid; i < C * (D / 8); i += kSimtThreads) {
      const int r = i / (D / 8), c = (i % (D / 8)) * 8;
      uint4 u = make_uint4(0u, 0u, 0u, 0u);
      if (r < n) u = __ldg(reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(src) + (tok_h + (size_t)r * H) * D + c));
      const uint32_t w[4] = {u.x, u.y, u.z, u.w};
      float f[8];
#pragma unroll
      for (int e = 0; e < 4; ++e) { f[2 * e] = __uint_as_float(w[e] << 16); f[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u); }
      *reinterpret_cast<float4*>(tile + r * (D + 4) + c) = make_float4(f[0], f[1], f[2], f[3]);
      *reinterpret_cast<float4*>(tile + r * (D + 4) + c + 4) = make_float4(f[4], f[5], f[6], f[7]);
    }
  };
  load_io_rows(std::integral_constant<int, DV>{}, Do, a.d_o, a.do_bf16);
  load_io_rows(std::integral_constant<int, DK>{}, Qs, a.q, a.in_bf16);
  load_io_rows(std::integral_constant<int, DK>{}, Ks, a.k, a.in_bf16);
  load_rows<DV>(Dr, nullptr, a.dr + tok_h * DV, false, (size_t)H * DV, n, tid);
  load_rows<DV>(Vt, nullptr, a.vt + slot_h * C * DV, false, DV, C, tid);
  fetch(0);
  fetch(1);

  // ---- vectors: the chain's coefficients, the gates, zeroed adjoints
  const float* cf = a.coef + slot_h * MDN_NUM_COEF * C;
  for (int i = tid; i < 24 * C; i += kSimtThreads) vec[i] = 0.f;
  __syncthreads();
  if (tid < C) {
    const int r = tid;
    V(vAbar)[r] = cf[kAbar * C + r]; V(vB)[r] = cf[kB * C + r]; V(vP)[r] = cf[kAlphaBPrev * C + r];
    V(vGS)[r] = cf[kGS * C + r]; V(vGM)[r] = cf[kGM * C + r]; V(vMubar)[r] = cf[kMubar * C + r];
    V(vAlpha)[r] = cf[kAlpha * C + r]; V(vMu)[r] = cf[kMu * C + r]; V(vBeta)[r] = cf[kBeta * C + r]; V(vEta)[r] = cf[kEta * C + r];
    V(vBprev)[r] = r > 0 ? cf[kB * C + r - 1] : 0.f;
  }
  {   // the end-of-chunk adjoints d mubar_C = <dM', M>, d abar_C = <dS', S>, d b_C = -<dS', M>
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll 4
    for (int i = tid; i < DK * DV / 4; i += kSimtThreads) {
      const float4 S = __ldg(reinterpret_cast<const float4*>(fS) + i), M = __ldg(reinterpret_cast<const float4*>(fS + DK * DV) + i);
      const float4 dS = __ldg(reinterpret_cast<const float4*>(aS) + i), dM = __ldg(reinterpret_cast<const float4*>(aS + DK * DV) + i);
      s0 = fmaf(dM.x, M.x, fmaf(dM.y, M.y, fmaf(dM.z, M.z, fmaf(dM.w, M.w, s0))));
      s1 = fmaf(dS.x, S.x, fmaf(dS.y, S.y, fmaf(dS.z, S.z, fmaf(dS.w, S.w, s1))));
      s2 = fmaf(dS.x, M.x, fmaf(dS.y, M.y, fmaf(dS.z, M.z, fmaf(dS.w, M.w, s2))));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, off);
      s1 += __shfl_xor_sync(0xffffffffu, s1, off);
      s2 += __shfl_xor_sync(0xffffffffu, s2, off);
    }
    if (lane == 0) {
      atomicAdd(V(vdMubar) + n - 1, s0);
      atomicAdd(V(vdAbar) + n - 1, s1);
      atomicAdd(V(vdB) + n - 1, -s2);
    }
  }

  float2 dQ[4][E2], dK[4][E2];
  zero2(dQ); zero2(dK);
  int p = 0;
  // one pass: G = A B^T against the next state of the ring;  acc += w.G;  a coefficient vector's adjoint += sign sum_d G o X
  auto pass = [&](const float* A, float2 (&acc)[4][E2], const float* w, float wf, const float* X, float* dvec, float sign) {
    float2 G[4][2 * E2];
    zero2(G);
#pragma unroll 1
    for (int jb = 0; jb < NP; ++jb, ++p) {
      cp_wait<1>();
      __syncthreads();   // piece p is in; piece p - 1 has been read: its stage takes p + 2
      fetch(p + 2);
      dot_tile<4, 2 * E2>(G, A + rl * LDV + jb * 32, 16 * LDV, sm + L::st + (p % L::kStages) * L::kStage + dg * LB, 16 * LB, 0, 8);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = rl + 16 * i;
      const float wr = wf * w[r];
      float s = 0.f;
#pragma unroll
      for (int e = 0; e < E2; ++e) {
        const float2 g = make_float2(hsum(G[i][e]), hsum(G[i][e + E2]));
        const float2 x = *reinterpret_cast<const float2*>(X + r * LDK + 2 * dg + 32 * e);
        acc[i][e] = __ffma2_rn(make_float2(wr, wr), g, acc[i][e]);
        s = fmaf(g.x, x.x, fmaf(g.y, x.y, s));
      }
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      s += __shfl_xor_sync(0xffffffffu, s, 4);
      if ((tid & 7) == 0) atomicAdd(dvec + r, sign * s);
    }
  };
  pass(Do, dQ, V(vAbar), scale, Qs, V(vdAbar), scale);     // dO S^T
  pass(Do, dQ, V(vB), -scale, Qs, V(vdB), -scale);         // dO M^T
  pass(Dr, dK, V(vAbar), -1.f, Ks, V(vdAbar), -1.f);       // dR S^T
  pass(Dr, dK, V(vP), 1.f, Ks, V(vdP), 1.f);               // dR M^T
  pass(Vt, dK, V(vGS), 1.f, Ks, V(vdGS), 1.f);             // V~ dS'^T
  pass(Vt, dK, V(vGM), -1.f, Ks, V(vdGM), -1.f);           // V~ dM'^T
  cp_wait<0>();
  __syncthreads();   // the ring has been read: gamma, m take its place

  if (tid < C) {          // gamma by the column recurrence of Eq. 10 (thread = column), zero above the diagonal
    const int i = tid;
    float m = 1.f, gam = 0.f;
#pragma unroll 4
    for (int r = 0; r < C; ++r) {
      if (r > i) m *= V(vMu)[r];
      if (r >= i) gam = fmaf(V(vAlpha)[r], gam, V(vBeta)[r] * m);
      Gam[r * kLT + i] = r >= i ? gam : 0.f;
    }
  } else if (tid < 2 * C) {   // m_{r,i} = mu_{i+1} .. mu_r
    const int i = tid - C;
    float m = 1.f;
#pragma unroll 4
    for (int r = 0; r < C; ++r) {
      if (r > i) m *= V(vMu)[r];
      Mm[r * kLT + i] = r >= i ? m : 0.f;
    }
  }
  // ---- the four 64 x 64 products, lower triangle in 16 x 16 blocks: rows rl + 16 i, columns dg + 16 e, e <= i
  auto product = [&](float (&out)[4][4], const float* A, int lda, const float* B, int ldb, int K) {
    float2 acc[4][4];
    zero2(acc);
#pragma unroll 1
    for (int k = 0; k < K; k += 4) {
      float4 av[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = lds4(A + (rl + 16 * i) * lda + k);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float4 bv = lds4(B + (dg + 16 * e) * ldb + k);
#pragma unroll
        for (int i = e; i < 4; ++i) fma4(acc[i][e], av[i], bv);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) out[i][e] = hsum(acc[i][e]);
  };
  float P1[4][4], P2[4][4], QK[4][4], KK[4][4];
  product(P1, Do, LDV, Vt, LDV, DV);      // dO V~^T
  product(P2, Dr, LDV, Vt, LDV, DV);      // dR V~^T
  product(QK, Qs, LDK, Ks, LDK, DK);
  product(KK, Ks, LDK, Ks, LDK, DK);
  __syncthreads();   // dO, dR, V~ have been read; gamma, m complete
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int r = rl + 16 * i, c = dg + 16 * e;
      const float dOVt = (r < n && c <= r) ? P1[i][e] : 0.f;
      const float dA = (r < n && c < r) ? -P2[i][e] : 0.f;
      const float et = V(vEta)[c];
      const float dw = scale * Gam[r * kLT + c] * et * dOVt;
      const float da = (r > 0 ? V(vAlpha)[r] * Gam[(r - 1) * kLT + c] * et : 0.f) * dA;
      DW[r * kLT + c] = dw;
      DWT[c * kLT + r] = dw;
      if (c < r) { DAS[r * kLT + c] = da; DAS[c * kLT + r] = da; }
      else if (c == r) DAS[r * kLT + r] = 0.f;
      dGe[r * kLT + c] = scale * dOVt * QK[i][e];
      dGm[r * kLT + c] = dA * KK[i][e];
    }
  __syncthreads();
  // ---- dQ += DW K;  dK += DW^T Q + (DA + DA^T) K
  auto rows_times = [&](float2 (&acc)[4][E2], const float* A, const float* B) {
#pragma unroll 1
    for (int k = 0; k < n; k += 4) {
      float4 av[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = lds4(A + (rl + 16 * i) * kLT + k);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float2 b[E2];
#pragma unroll
        for (int e = 0; e < E2; ++e) b[e] = *reinterpret_cast<const float2*>(B + (k + u) * LDK + 2 * dg + 32 * e);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float x = u == 0 ? av[i].x : u == 1 ? av[i].y : u == 2 ? av[i].z : av[i].w;
#pragma unroll
          for (int e = 0; e < E2; ++e) acc[i][e] = __ffma2_rn(make_float2(x, x), b[e], acc[i][e]);
        }
      }
    }
  };
  rows_times(dQ, DW, Ks);
  rows_times(dK, DWT, Qs);
  rows_times(dK, DAS, Ks);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = rl + 16 * i;
    if (r < n) {
#pragma unroll
      for (int e = 0; e < E2; ++e) {
        const size_t at = (tok_h + (size_t)r * H) * DK + 2 * dg + 32 * e;
        *reinterpret_cast<float2*>(a.dq + at) = dQ[i][e];
        *reinterpret_cast<float2*>(a.dk + at) = dK[i][e];
      }
    }
  }
  __syncthreads();   // DW, DW^T, DA have been read: the gate gradients' work matrices take their places
  gate_gradients(vec, GateMats{Gam, Mm, dGe, dGm, DW, DWT}, DAS, n, tok_h, H, a.gates);
}

template <int DK, int NV> cudaError_t launch_adj(const Plan& pl, const AdjArgs& a) {
  const size_t smem = AdjSmem<DK, NV>::bytes(a.in_bf16);
  const cudaError_t e = cudaFuncSetAttribute(adj_chain_kernel<DK, NV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(adj_chain_kernel<DK, NV>, dim3((unsigned)pl.geom.num_seqs * pl.p.H * (a.dv / NV)), dim3(kSimtThreads), smem,
                    pl.stream, a);
}
template <int DK, int DV> cudaError_t launch_par(const Plan& pl, const ParArgs& a) {
  constexpr size_t smem = (size_t)ParSmem<DK, DV>::kFloats * 4;
  const cudaError_t e = cudaFuncSetAttribute(bwd_exact_par_kernel<DK, DV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(bwd_exact_par_kernel<DK, DV>, dim3((unsigned)pl.geom.num_slots * pl.p.H), dim3(kSimtThreads), smem, pl.stream, a);
}

}  // namespace

void bwd_scratch_layout(const mdn_params& p, int num_slots, BwdScratch* s) {
  const uint64_t mats = (uint64_t)num_slots * p.H;
  uint64_t off = 0;
  auto take = [&](uint64_t floats) { const uint64_t at = off; off = (off + floats * 4 + 255) / 256 * 256; return at; };
  s->tt = take(mats * C * C);
  s->states = take(mats * 2 * p.dk * p.dv);
  s->adj = take(mats * 2 * p.dk * p.dv);
  s->vt = take(mats * C * p.dv);
  s->total = off;
}

cudaError_t launch_bwd_exact(const Plan& pl, const BwdIo& io, char* scratch, const BwdScratch& sl, int* launches) {
  float* tt = reinterpret_cast<float*>(scratch + sl.tt);
  float* states = reinterpret_cast<float*>(scratch + sl.states);
  float* adj = reinterpret_cast<float*>(scratch + sl.adj);
  float* vt = reinterpret_cast<float*>(scratch + sl.vt);
  cudaError_t e = launch_intra_simt(pl, io.q, io.k, GateArgs{io.beta, io.log_alpha, io.log_mu, io.eta}, tt, launches);
  if (e != cudaSuccess) return e;
  e = launch_chain_simt_keep(pl, io.k, io.v, io.S0, io.M0, states, vt, launches);
  if (e != cudaSuccess) return e;
  const bool in_bf16 = pl.p.io_dtype == MDN_BF16, do_bf16 = pl.p.o_dtype == MDN_BF16;
  const float* coef = reinterpret_cast<const float*>(pl.ws + pl.lay.off_coef);
  AdjArgs a{};
  a.g = pl.geom;
  a.q = io.q; a.k = io.k; a.d_o = io.d_o;
  a.in_bf16 = in_bf16; a.do_bf16 = do_bf16;
  a.dv = pl.p.dv;
  a.coef = coef; a.TT = tt; a.WT = reinterpret_cast<const float*>(pl.ws + pl.lay.off_W);
  a.dSf = io.dSf; a.dMf = io.dMf;
  a.scale = pl.p.scale;
  a.adj = adj; a.dv_out = io.dv;
  a.dS0 = io.dS0; a.dM0 = io.dM0;
  const bool narrow = simt_narrow_columns(pl);
  if (pl.p.dk == 64) e = narrow ? launch_adj<64, 8>(pl, a) : launch_adj<64, 16>(pl, a);
  else e = narrow ? launch_adj<128, 8>(pl, a) : launch_adj<128, 16>(pl, a);
  if (e != cudaSuccess) return e;
  ++*launches;
  ParArgs b{};
  b.g = pl.geom;
  b.q = io.q; b.k = io.k; b.d_o = io.d_o;
  b.in_bf16 = in_bf16; b.do_bf16 = do_bf16;
  b.coef = coef; b.states = states; b.adj = adj; b.vt = vt; b.dr = io.dv;
  b.scale = pl.p.scale;
  b.dq = io.dq; b.dk = io.dk;
  b.gates = GateOut{io.dbeta, io.dlog_alpha, io.dlog_mu, io.deta};
  if (pl.p.dk == 64) e = pl.p.dv == 64 ? launch_par<64, 64>(pl, b) : launch_par<64, 128>(pl, b);
  else e = pl.p.dv == 64 ? launch_par<128, 64>(pl, b) : launch_par<128, 128>(pl, b);
  if (e == cudaSuccess) ++*launches;
  return e;
}

}  // namespace mdn
