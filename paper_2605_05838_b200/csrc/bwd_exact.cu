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
// by the scans of Eq. 10 in reverse (bwd_gates.cuh).  Four kernels (packed input: the chunk map before them):
//   intra_simt (scan, T, T^T, W^T dO);  chain_simt without output terms (the states at every chunk's start, V~);
//   the adjoint chain (dS', dM' at every chunk's end, dR);  the per-chunk kernel (everything else, all chunks in parallel).
// Short sequences go token by token instead (bwd_short.cu, which holds the rule).
//
// Why: the serial part of a backward is two walks over the chunks.  The token-by-token form this replaces was serial
// over tokens (3.4 us per token and chain whatever the GPU's size: 3.4 ms for T = 1023, B H = 16); here 64 tokens cost
// one chunk step of either chain, and the bulk of the arithmetic (20 of 28 products) is parallel over chunks.
#include <type_traits>

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
  const float* coef; const float* TT;
  const float* vp;       // W^T dO, [slot][H][64][dv]
  const float* dSf; const float* dMf;
  float scale;
  float* adj;            // [slot][H][2][dk][dv]: dS', dM' at the chunk's end
  float* dv_out;         // dR = dL/dv, [B,T,H,dv]
  float* dS0; float* dM0;
  int short_limit;       // sequences of up to so many tokens are bwd_short.cu's
};

template <int DK, int NV> struct AdjSmem {   // float offsets
  static constexpr int LDK = DK + 4, LDW = 2 * NV + 4;
  static constexpr int K = 0, Q = K + 2 * C * LDK, TT = Q + C * LDK, D = TT + C * kLT, Zt = D + 2 * NV * LDK, Wd = Zt + NV * kLT,
                       cv = Wd + 2 * C * LDW, kFloats = cv + 2 * kChainCoefs * C;
  static constexpr size_t bytes(bool bf16) { return (size_t)kFloats * 4 + (bf16 ? (size_t)2 * C * DK * 2 : 0); }
};

// One CTA per (sequence, head, NV value columns), chunks from last to first; the columns of dS', dM' stay in shared
// memory.  The forward chain's structure and tiles (chain_simt.cu) with W^T dO in the place of V; the two Q terms make its
// state update twice as long (rows of K, then rows of Q).
template <int DK, int NV>
__global__ void __launch_bounds__(kChainThreads<NV>, 1) adj_chain_kernel(const AdjArgs a) {
  extern __shared__ __align__(16) float sm[];
  using L = AdjSmem<DK, NV>;
  constexpr int TH = kChainThreads<NV>, LDK = L::LDK, LDW = L::LDW;
  float* Qs = sm + L::Q;
  float* TTm = sm + L::TT;
  float* Ds = sm + L::D;       // [2 NV (columns of dS', then of dM')][LDK]
  float* Zt = sm + L::Zt;      // dV~^T
  float* Wd = sm + L::Wd;      // [128 rows (K, then Q)][LDW]: per column the weights of the update of dS', dM'
  uint8_t* raw = reinterpret_cast<uint8_t*>(sm + L::kFloats);
  uint8_t* rawQ = raw + C * DK * 2;

  const int tid = threadIdx.x;
  const StateTile<NV, 1> st_tile(tid);
  const TriTile<NV> tri(tid);
  const int H = a.g.H, DV = a.dv, NVB = DV / NV;
  const int vb = blockIdx.x % NVB, h = (blockIdx.x / NVB) % H, seq = blockIdx.x / (NVB * H);
  const int j0 = vb * NV;
  grid_dependency_wait();
  grid_launch_dependents();
  const SeqInfo sq = seq_info(a.g, seq);
  if (short_sequence(sq, a.short_limit)) return;
  const size_t st_off = ((size_t)seq * H + h) * DK * DV;
  const size_t es = a.in_bf16 ? 2 : 4;
  const int nch = sq.nchunks;
  auto src_of = [&](const void* p, int c) {
    return static_cast<const void*>(static_cast<const uint8_t*>(p) + ((size_t)(sq.tok0 + c * C) * H + h) * DK * es);
  };
  auto fetch_k = [&](int c) {
    load_rows<DK, TH>(sm + L::K + (c & 1) * C * LDK, raw, src_of(a.k, c), a.in_bf16, (size_t)H * DK, min(C, sq.len - c * C), tid);
    const float* cf = a.coef + ((size_t)(sq.slot0 + c) * H + h) * MDN_NUM_COEF * C;
    if (tid < kChainCoefs * C / 4) cp16(sm + L::cv + (c & 1) * kChainCoefs * C + tid * 4, cf + tid * 4, true);
  };
  auto mat = [&](int c) { return ((size_t)(sq.slot0 + c) * H + h) * C * C; };

  if (nch > 0) {
    fetch_k(nch - 1);
    load_mat<TH>(TTm, a.TT + mat(nch - 1), tid);
    cp_commit();
  }
  for (int i = tid; i < 2 * NV * DK; i += TH) {
    const int jj = i % NV, d = (i / NV) % DK, which = i / (NV * DK);
    const float* src = which ? a.dMf : a.dSf;
    Ds[(which * NV + jj) * LDK + d] = src ? src[st_off + (size_t)d * DV + j0 + jj] : 0.f;
  }

  for (int c = nch - 1; c >= 0; --c) {
    const int n = min(C, sq.len - c * C);
    const size_t slot_h = (size_t)(sq.slot0 + c) * H + h, tok_h = (size_t)(sq.tok0 + c * C) * H + h;
    float* Ks = sm + L::K + (c & 1) * C * LDK;
    const float* cv = sm + L::cv + (c & 1) * kChainCoefs * C;
    float vp[st_tile.kPairs], dox[16 / tri.SL];
    st_tile.own([&](int e, int, int r, int j) { vp[e] = __ldg(a.vp + (slot_h * C + r) * DV + j0 + j); });
    tri.own([&](int e, int r, int j) { dox[e] = r < n ? load_io(a.d_o, (tok_h + (size_t)r * H) * DV + j0 + j, a.do_bf16) : 0.f; });
    cp_wait<0>();
    __syncthreads();   // tiles landed; the previous step's readers are done, its adjoints are written
    if (a.in_bf16) {
      widen_tile<DK, TH>(Ks, raw, tid);
      __syncthreads();
    }
    if (c > 0) fetch_k(c - 1);
    load_rows<DK, TH>(Qs, rawQ, src_of(a.q, c), a.in_bf16, (size_t)H * DK, n, tid);
    cp_commit();
    {   // the adjoint pair at the chunk's end, [d][j]
      float* dst = a.adj + slot_h * 2 * DK * DV + j0;
      for (int i = tid; i < 2 * NV * DK; i += TH) {
        const int j = i % NV, d = (i / NV) % DK, which = i / (NV * DK);
        dst[(size_t)which * DK * DV + (size_t)d * DV + j] = Ds[(which * NV + j) * LDK + d];
      }
    }
    tri.own([&](int e, int r, int j) {   // weights of the Q rows
      *reinterpret_cast<float2*>(Wd + (C + r) * LDW + 2 * j) = make_float2(a.scale * cv[kAbar * C + r] * dox[e], -a.scale * cv[kB * C + r] * dox[e]);
    });

    // ---- 1: dV~ = W^T dO + g_S.(K dS') - g_M.(K dM')
    st_tile.template run<DK>(Ks, Ks, Ds, [&](int e, int, int r, int j, float xs, float xm) {
      Zt[j * kLT + r] = vp[e] + cv[kGS * C + r] * xs - cv[kGM * C + r] * xm;
    });
    __syncthreads();

    // ---- 2: dR = T^T dV~  (upper triangular)
    tri.template run<false>(TTm, Zt, [&](int r, int j, float x) {
      if (r < n) a.dv_out[(tok_h + (size_t)r * H) * DV + j0 + j] = x;
      *reinterpret_cast<float2*>(Wd + r * LDW + 2 * j) = make_float2(-cv[kAbar * C + r] * x, cv[kAlphaBPrev * C + r] * x);
    });
    cp_wait<0>();   // Q (and K of the next step) are in
    __syncthreads();
    if (a.in_bf16) {
      widen_tile<DK, TH>(Qs, rawQ, tid);
      __syncthreads();
    }
    if (c > 0) load_mat<TH>(TTm, a.TT + mat(c - 1), tid);   // T^T has been read
    cp_commit();

    // ---- 3: the adjoint pair at the chunk's start (one owner per entry)
    {
      UpdateTile<DK, NV> up(tid);
      up.add(Ks, Wd, n);
      up.add(Qs, Wd + C * LDW, n);
      const float aC = cv[kAbar * C + C - 1], bC = cv[kB * C + C - 1], mC = cv[kMubar * C + C - 1];
      up.finish([&](int d, int j, float ds, float dm) {
        float* sp = Ds + j * LDK + d;
        float* mp = sp + NV * LDK;
        const float s = *sp, m = *mp;
        *sp = aC * s + ds;
        *mp = mC * m - bC * s + dm;
      });
    }
  }
  cp_wait<0>();
  __syncthreads();
  for (int i = tid; i < 2 * NV * DK; i += TH) {
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
  int short_limit;
};

template <int DK, int DV> struct ParSmem {   // float offsets
  static constexpr int LDK = DK + 4, LDV = DV + 4, kMat = C * kLT;
  static constexpr int kStages = 3, kStage = DK * 32, kStageArea = kStages * kStage;
  static constexpr int K = 0, Q = K + C * LDK, vec = Q + C * LDK, st = vec + 24 * C, tiles = st + kStageArea,
                       kTiles = 3 * C * LDV > 5 * kMat ? 3 * C * LDV : 5 * kMat, kFloats = tiles + kTiles;
  static_assert(kFloats * 4 <= 232448 && kStageArea >= kMat && kMat >= kGateScratch, "shared memory");
};

// One 256-thread CTA per (chunk, head); its two halves of 128 threads work on different products of the same step, each
// thread on 8 rows x dk / 16 columns (simt_tile.cuh: the tile that balances operand loads and FMAs):
//   half 0:  V~ dS'^T (a part of dK),  dO S^T, dO M^T (dQ),   dO V~^T, Q K^T,  DW K
//   half 1:  V~ dM'^T, dR S^T, dR M^T (dK),                                 dR V~^T, K K^T,  DW^T Q, (DA + DA^T) K
// The states stream through a three-stage ring (32 value columns of S or M, or 16 of dS' and dM' each); dO, dR, V~, K, Q stay in
// shared memory.  Chunks of up to 32 tokens take tiles of 4 rows.  Bound by the fp32 pipes and the
// shared-memory port alike: 9.5 M multiply-adds per chunk and head at dk = dv = 128.
template <int DK, int DV>
__global__ void __launch_bounds__(kSimtThreads, 1) bwd_exact_par_kernel(const ParArgs a) {
  extern __shared__ __align__(16) float sm[];
  using L = ParSmem<DK, DV>;
  constexpr int LDK = L::LDK, LDV = L::LDV, E2 = DK / 32, NP = DV / 32;
  float* Ks = sm + L::K;
  float* Qs = sm + L::Q;
  float* vec = sm + L::vec;
  float* Do = sm + L::tiles;
  float* Dr = Do + C * LDV;
  float* Vt = Dr + C * LDV;
  // after the streams / the products: 64 x 64 matrices
  float* Gam = sm + L::st;
  float* DW = sm + L::tiles;
  float* DWT = DW + L::kMat;
  float* DAS = DWT + L::kMat;   // DA + DA^T
  float* dGe = DAS + L::kMat;
  float* dGm = dGe + L::kMat;
  auto V = [&](int which) { return vec + which * C; };

  const int H = a.g.H, slot = blockIdx.x / H, h = blockIdx.x % H;
  grid_dependency_wait();
  grid_launch_dependents();
  const SlotInfo si = slot_info(a.g, slot);
  if (si.seq < 0 || short_sequence(si, a.short_limit)) return;
  const int n = si.n;
  const int tid = threadIdx.x, lane = tid & 31;
  const bool half1 = tid >= 128;
  const int dg = tid & 15, rl = (tid >> 4) & 7;   // columns 2 dg + 32 e (+ 1), rows rl + 8 i
  const size_t slot_h = (size_t)slot * H + h, tok_h = (size_t)si.tok0 * H + h;
  const float* fS = a.states + slot_h * 2 * DK * DV;
  const float* aS = a.adj + slot_h * 2 * DK * DV;
  const float scale = a.scale;

  // ---- the ring.  Key row d of a state lies at ring row p(d) = (d & 1) dk / 2 + d / 2, so that a thread's column PAIRS are rows
  // dg + 16 e of either half; the 16-byte pieces of a row are XOR-swizzled with the row: conflict-free loads
  auto fetch = [&](int step) {
    if (step < 4 * NP) {
      float* dst = sm + L::st + (step % L::kStages) * L::kStage;
      const bool adj = step < 2 * NP;
      const float* src = adj ? aS + step * 16 : fS + (step < 3 * NP ? (step - 2 * NP) * 32 : (size_t)DK * DV + (step - 3 * NP) * 32);
#pragma unroll
      for (int i = 0; i < DK * 8 / kSimtThreads; ++i) {
        const int idx = tid + i * kSimtThreads;
        if (adj) {   // dS' rows, then dM' rows, four pieces each
          const int which = idx / (DK * 4), d = (idx >> 2) % DK, u = idx & 3, p = (d & 1) * (DK / 2) + (d >> 1);
          cp16(dst + (which * DK + p) * 16 + ((u ^ (p >> 1)) & 3) * 4, src + (size_t)which * DK * DV + (size_t)d * DV + u * 4, true);
        } else {
          const int d = idx >> 3, u = idx & 7, p = (d & 1) * (DK / 2) + (d >> 1);
          cp16(dst + p * 32 + ((u ^ p) & 7) * 4, src + (size_t)d * DV + u * 4, true);
        }
      }
    }
    cp_commit();
  };
  auto head = [&](const void* p, bool bf16, int D) { return static_cast<const void*>(static_cast<const uint8_t*>(p) + tok_h * D * (bf16 ? 2 : 4)); };
  load_rows<DV>(Vt, nullptr, a.vt + slot_h * C * DV, false, DV, C, tid);
  load_io_rows(Ks, head(a.k, a.in_bf16, DK), a.in_bf16, DK, (size_t)H * DK, n, tid);
  fetch(0);
  load_io_rows(Do, head(a.d_o, a.do_bf16, DV), a.do_bf16, DV, (size_t)H * DV, n, tid);
  load_io_rows(Qs, head(a.q, a.in_bf16, DK), a.in_bf16, DK, (size_t)H * DK, n, tid);
  load_rows<DV>(Dr, nullptr, a.dr + tok_h * DV, false, (size_t)H * DV, n, tid);
  fetch(1);

  // ---- vectors: the chain's coefficients, the gates, zeroed adjoints
  const float* cf = a.coef + slot_h * MDN_NUM_COEF * C;
  for (int i = tid; i < 24 * C; i += kSimtThreads) vec[i] = 0.f;
  __syncthreads();
  if (tid < C) {   // (all loads before the first store: they must not wait for one another)
    const int r = tid;
    auto ld = [&](int which, int at) { return __ldg(cf + which * C + at); };
    const float x0 = ld(kAbar, r), x1 = ld(kB, r), x2 = ld(kAlphaBPrev, r), x3 = ld(kGS, r), x4 = ld(kGM, r), x5 = ld(kMubar, r);
    const float x6 = ld(kAlpha, r), x7 = ld(kMu, r), x8 = ld(kBeta, r), x9 = ld(kEta, r), x10 = ld(kB, max(r - 1, 0));
    V(vAbar)[r] = x0; V(vB)[r] = x1; V(vP)[r] = x2; V(vGS)[r] = x3; V(vGM)[r] = x4; V(vMubar)[r] = x5;
    V(vAlpha)[r] = x6; V(vMu)[r] = x7; V(vBeta)[r] = x8; V(vEta)[r] = x9;
    V(vBprev)[r] = r > 0 ? x10 : 0.f;
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

  auto body = [&](auto rows_tag) {
    constexpr int R = decltype(rows_tag)::value;   // rows rl + 8 i, i < R, cover the chunk's n tokens
    int step = 0;
    // dQ (half 0) and dK (half 1) are summed in their places in global memory (L2): the accumulators of one product are all
    // the registers can hold next to operands that are on their way
    auto at = [&](float* g, int r, int e) { return reinterpret_cast<float2*>(g + (tok_h + (size_t)r * H) * DK + 2 * dg + 32 * e); };
    // G = A B^T over the next `steps` stages of the ring (cols = 16 or 32 value columns each); a coefficient vector's adjoint
    // += sign (row sums of G o X).  G's column pairs are left in G[i][e].x, G[i][e + E2].x.
    auto product = [&](const float* A, int steps, auto cols_tag, const float* X, float* dvec, float sign, auto& G) {
      constexpr int kCols = decltype(cols_tag)::value;
      zero2(G);
      const int swz = kCols == 16 ? (dg >> 1) & 3 : dg & 7;
#pragma unroll 1
      for (int jb = 0; jb < steps; ++jb, ++step) {
        cp_wait<1>();
        __syncthreads();   // this step's stage is in; the previous step's has been read and takes step + 2
        fetch(step + 2);
        const float* b0 = sm + L::st + (step % L::kStages) * L::kStage + (kCols == 16 && half1 ? DK * 16 : 0) + dg * kCols;
        const float* a0 = A + rl * LDV + jb * kCols;
#pragma unroll 2
        for (int k = 0; k < kCols / 4; ++k) {
          float4 av[R];
#pragma unroll
          for (int i = 0; i < R; ++i) av[i] = lds4(a0 + 8 * i * LDV + 4 * k);
#pragma unroll
          for (int e = 0; e < 2 * E2; ++e) {
            const float4 bv = lds4(b0 + 16 * e * kCols + ((k ^ swz) << 2));
#pragma unroll
            for (int i = 0; i < R; ++i) fma4(G[i][e], av[i], bv);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const int r = rl + 8 * i;
        float s = 0.f;
#pragma unroll
        for (int e = 0; e < E2; ++e) {
          const float2 g = make_float2(hsum(G[i][e]), hsum(G[i][e + E2]));
          const float2 x = *reinterpret_cast<const float2*>(X + r * LDK + 2 * dg + 32 * e);
          s = fmaf(g.x, x.x, fmaf(g.y, x.y, s));
          G[i][e] = g;
        }
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        s += __shfl_xor_sync(0xffffffffu, s, 4);
        s += __shfl_xor_sync(0xffffffffu, s, 8);
        if (dg == 0) atomicAdd(dvec + r, sign * s);
      }
    };
    // dst (+)= w_r G
    auto put = [&](float* dst, float wf, const float* w, const auto& G, bool onto) {
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const int r = rl + 8 * i;
        if (r < n) {
          const float wr = wf * w[r];
          float2 x[E2];
#pragma unroll
          for (int e = 0; e < E2; ++e) x[e] = onto ? *at(dst, r, e) : make_float2(0.f, 0.f);
#pragma unroll
          for (int e = 0; e < E2; ++e) *at(dst, r, e) = __ffma2_rn(make_float2(wr, wr), G[i][e], x[e]);
        }
      }
    };
    {
      float2 G[R][2 * E2];
      product(Vt, 2 * NP, std::integral_constant<int, 16>{}, Ks, V(half1 ? vdGM : vdGS), half1 ? -1.f : 1.f, G);
      if (!half1) put(a.dk, 1.f, V(vGS), G, false);
      __syncthreads();   // half 0's part of dK is there; from here on half 1 alone adds to it
      if (half1) put(a.dk, -1.f, V(vGM), G, true);
    }
    const float* A = half1 ? Dr : Do;
    const float* X = half1 ? Ks : Qs;
    float* dst = half1 ? a.dk : a.dq;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {   // against S, against M
      float2 G[R][2 * E2];
      const float w = (half1 ? -1.f : scale) * (pass ? -1.f : 1.f);
      product(A, NP, std::integral_constant<int, 32>{}, X, V(pass == 0 ? vdAbar : half1 ? vdP : vdB), w, G);
      put(dst, w, V(pass == 0 ? vAbar : half1 ? vP : vB), G, half1 || pass > 0);
    }
    cp_wait<0>();
    __syncthreads();   // the ring has been read: gamma takes its place

    if (tid < C) {          // gamma by the column recurrence of Eq. 10 (thread = column), zero above the diagonal
      const int i = tid;
      float m = 1.f, gam = 0.f;
#pragma unroll 4
      for (int r = 0; r < C; ++r) {
        if (r > i) m *= V(vMu)[r];
        if (r >= i) gam = fmaf(V(vAlpha)[r], gam, V(vBeta)[r] * m);
        Gam[r * kLT + i] = r >= i ? gam : 0.f;
      }
    }
    // ---- the four 64 x 64 products, lower triangle: rows rl + 8 i, columns dg + 16 e, e <= i / 2
    auto square = [&](float (&out)[R][4], const float* A, int lda, const float* B, int ldb, int K) {
      float2 t[R][4];
      zero2(t);
#pragma unroll 1
      for (int k = 0; k < K; k += 4) {
        float4 av[R];
#pragma unroll
        for (int i = 0; i < R; ++i) av[i] = lds4(A + (rl + 8 * i) * lda + k);
#pragma unroll
        for (int e = 0; e < (R + 1) / 2; ++e) {
          const float4 bv = lds4(B + (dg + 16 * e) * ldb + k);
#pragma unroll
          for (int i = 2 * e; i < R; ++i) fma4(t[i][e], av[i], bv);
        }
      }
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) out[i][e] = hsum(t[i][e]);
    };
    float P[R][4], XK[R][4];
    square(P, A, LDV, Vt, LDV, DV);      // dO V~^T | dR V~^T
    square(XK, X, LDK, Ks, LDK, DK);     // Q K^T   | K K^T
    __syncthreads();   // dO, dR, V~ have been read; gamma complete
    // (rows past the tiles' reach: the matrices' rows and columns there are cleared for the gate gradients below)
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int r = rl + 8 * i, c = dg + 16 * e;
        const float et = V(vEta)[c];
        const float p = i < R ? P[i < R ? i : 0][e] : 0.f, xk = i < R ? XK[i < R ? i : 0][e] : 0.f;
        if (!half1) {
          const float dOVt = (r < n && c <= r) ? p : 0.f;
          const float dw = scale * Gam[r * kLT + c] * et * dOVt;
          DW[r * kLT + c] = dw;
          DWT[c * kLT + r] = dw;
          dGe[r * kLT + c] = scale * dOVt * xk;
        } else {
          const float dA = (r < n && c < r) ? -p : 0.f;
          const float da = (r > 0 ? V(vAlpha)[r] * Gam[(r - 1) * kLT + c] * et : 0.f) * dA;
          if (c < r) { DAS[r * kLT + c] = da; DAS[c * kLT + r] = da; }
          else if (c == r) DAS[r * kLT + r] = 0.f;
          dGm[r * kLT + c] = dA * xk;
        }
      }
    __syncthreads();
    // ---- dQ += DW K;  dK += DW^T Q + (DA + DA^T) K
    float2 acc[R][E2];
    zero2(acc);
    auto rows_times = [&](const float* A, const float* B) {
#pragma unroll 1
      for (int k = 0; k < n; k += 4) {
        float4 av[R];
#pragma unroll
        for (int i = 0; i < R; ++i) av[i] = lds4(A + (rl + 8 * i) * kLT + k);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          float2 b[E2];
#pragma unroll
          for (int e = 0; e < E2; ++e) b[e] = *reinterpret_cast<const float2*>(B + (k + u) * LDK + 2 * dg + 32 * e);
#pragma unroll
          for (int i = 0; i < R; ++i) {
            const float x = u == 0 ? av[i].x : u == 1 ? av[i].y : u == 2 ? av[i].z : av[i].w;
#pragma unroll
            for (int e = 0; e < E2; ++e) acc[i][e] = __ffma2_rn(make_float2(x, x), b[e], acc[i][e]);
          }
        }
      }
    };
    rows_times(half1 ? DWT : DW, half1 ? Qs : Ks);
    if (half1) rows_times(DAS, Ks);
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = rl + 8 * i;
      if (r < n) {
#pragma unroll
        for (int e = 0; e < E2; ++e) {
          float2* to = at(dst, r, e);
          const float2 x = *to;
          *to = make_float2(x.x + acc[i][e].x, x.y + acc[i][e].y);
        }
      }
    }
  };
  if (n > 32) body(std::integral_constant<int, 8>{});
  else body(std::integral_constant<int, 4>{});
  __syncthreads();   // DW has been read: the gate gradients' scratch takes its place
  gate_gradients(vec, [&](int r, int i) { return dGe[r * kLT + i]; }, [&](int i) { return dGe[i * kLT + i]; }, [&](int r, int i) { return dGm[r * kLT + i]; }, DW, n, tok_h, H,
                 a.gates);
}

template <int DK, int NV> cudaError_t launch_adj(const Plan& pl, const AdjArgs& a) {
  const size_t smem = AdjSmem<DK, NV>::bytes(a.in_bf16);
  const cudaError_t e = allow_smem<(int)AdjSmem<DK, NV>::bytes(true)>(adj_chain_kernel<DK, NV>);
  if (e != cudaSuccess) return e;
  return launch_pdl(adj_chain_kernel<DK, NV>, dim3((unsigned)pl.geom.num_seqs * pl.p.H * (a.dv / NV)), dim3(kChainThreads<NV>), smem,
                    pl.stream, a);
}
template <int DK, int DV> cudaError_t launch_par(const Plan& pl, const ParArgs& a) {
  constexpr size_t smem = (size_t)ParSmem<DK, DV>::kFloats * 4;
  const cudaError_t e = allow_smem<(int)smem>(bwd_exact_par_kernel<DK, DV>);
  if (e != cudaSuccess) return e;
  return launch_pdl(bwd_exact_par_kernel<DK, DV>, dim3((unsigned)pl.geom.num_slots * pl.p.H), dim3(kSimtThreads), smem, pl.stream, a);
}

}  // namespace

void bwd_scratch_layout(const mdn_params& p, int num_slots, bool allow_short, BwdScratch* s) {
  s->shorts = allow_short ? bwd_short_plan(p) : BwdShort{-1, 0, 0};
  s->chunks = p.T > s->shorts.limit;
  const uint64_t mats = s->chunks ? (uint64_t)num_slots * p.H : 0;
  uint64_t off = 0;
  auto take = [&](uint64_t floats) { const uint64_t at = off; off = (off + floats * 4 + 255) / 256 * 256; return at; };
  s->tt = take(mats * C * C);
  s->states = take(mats * 2 * p.dk * p.dv);
  s->adj = take(mats * 2 * p.dk * p.dv);
  s->vt = take(mats * C * p.dv);
  s->vp = take(mats * C * p.dv);
  s->tokens = take(s->shorts.scratch_bytes / 4);
  s->total = off;
}

cudaError_t launch_bwd_exact(const Plan& pl, const BwdIo& io, char* scratch, const BwdScratch& sl, int* launches) {
  float* tt = reinterpret_cast<float*>(scratch + sl.tt);
  float* states = reinterpret_cast<float*>(scratch + sl.states);
  float* adj = reinterpret_cast<float*>(scratch + sl.adj);
  float* vt = reinterpret_cast<float*>(scratch + sl.vt);
  float* vp = reinterpret_cast<float*>(scratch + sl.vp);
  const int limit = sl.shorts.limit;
  if (limit >= 0) {
    const cudaError_t es = launch_bwd_short(pl, io, sl.shorts, scratch + sl.tokens, launches);
    if (es != cudaSuccess || !sl.chunks) return es;
  }
  cudaError_t e = launch_intra_simt(pl, io.q, io.k, GateArgs{io.beta, io.log_alpha, io.log_mu, io.eta}, IntraBwd{io.d_o, tt, vp, limit}, launches);
  if (e != cudaSuccess) return e;
  e = launch_chain_simt_keep(pl, io.k, io.v, io.S0, io.M0, states, vt, limit, launches);
  if (e != cudaSuccess) return e;
  const bool in_bf16 = pl.p.io_dtype == MDN_BF16, do_bf16 = pl.p.o_dtype == MDN_BF16;
  const float* coef = reinterpret_cast<const float*>(pl.ws + pl.lay.off_coef);
  AdjArgs a{};
  a.g = pl.geom;
  a.q = io.q; a.k = io.k; a.d_o = io.d_o;
  a.in_bf16 = in_bf16; a.do_bf16 = do_bf16;
  a.dv = pl.p.dv;
  a.coef = coef; a.TT = tt; a.vp = vp;
  a.dSf = io.dSf; a.dMf = io.dMf;
  a.scale = pl.p.scale;
  a.adj = adj; a.dv_out = io.dv;
  a.dS0 = io.dS0; a.dM0 = io.dM0;
  a.short_limit = limit;
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
  b.short_limit = limit;
  if (pl.p.dk == 64) e = pl.p.dv == 64 ? launch_par<64, 64>(pl, b) : launch_par<64, 128>(pl, b);
  else e = pl.p.dv == 64 ? launch_par<128, 64>(pl, b) : launch_par<128, 128>(pl, b);
  if (e == cudaSuccess) ++*launches;
  return e;
}

}  // namespace mdn
