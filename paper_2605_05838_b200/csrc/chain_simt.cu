// a3 + a4 in fp32 (any i/o type, dk, dv in {64, 128}): one CTA walks the chunks of one (sequence, head, block of NV
// value columns) in order, carrying its columns of S and M in shared memory.
//
// Per chunk (state equations and Eq. 11-12 of Section 3.1, in the form that applies T once):
//   R   = V - Diag(abar) (K S) + Diag(alpha b^-) (K M)          right-hand side of the solve
//   V~  = T R                                                    (T from the intra-chunk stage)
//   O   = scale (Diag(abar) (Q S) - Diag(b) (Q M)) + W V~        (W carries scale, Gamma, eta)
//   S' = abar_C S - b_C M + K^T Diag(gamma_C eta) V~
//   M' = mubar_C M - K^T Diag((mubar_C/mubar) eta) V~
// This equals the paper's U - Y S + Z M because T is linear and alpha_r abar_{r-1} = abar_r.
// Columns of S, M, V, V~, O never mix, so value-column blocks are independent CTAs.
//
// kOut = false is the forward sweep of the exact backward (bwd_exact.cu): no output terms; the states at every chunk's
// start and V~ go to global memory.
//
// What bounds it: the chunks are serial, so a chunk's latency is the kernel's time: 4 (NV = 8) or 8 products of a few
// thousand FMAs per thread-block between three barriers.  Hence NV is small (8 columns while that fills the SMs no more than
// once, else 16), every product is a register tile on packed FMAs (simt_tile.cuh), and the next chunk's K, Q, T, W are
// fetched by cp.async into buffers as they fall free (K twice buffered: it is the first and the last operand of a
// chunk).  Measured, B=1 H=2 T=256 dk=dv=64 (4 chunks) and the previous form (32 columns, one FMA per two shared-memory
// loads, loads exposed): see the table of cases in the design notes' performance section.
#include "simt_tile.cuh"

namespace mdn {
namespace {

struct ChainArgs {
  ChunkGeom g;
  const void* q; const void* k; const void* v;
  bool in_bf16, o_bf16;
  int dv;
  const float* coef; const float* T; const float* W;
  const float* S0; const float* M0;
  float scale;
  void* o;
  float* Sf; float* Mf;
  float* keep_states;   // kOut = false: [slot][H][2][dk][dv]
  float* keep_vt;       //               [slot][H][64][dv]
};

template <int DK, int NV> struct ChainSmem {   // float offsets
  static constexpr int LDK = DK + 4, LO = NV == 8 ? 8 : NV + 8;
  static constexpr int K = 0, St = K + 2 * C * LDK, T = St + 2 * NV * LDK, Rt = T + C * kLT, Wd = Rt + NV * kLT,
                       cv = Wd + C * NV * 4, kState = cv + 2 * kChainCoefs * C;
  static constexpr int Q = kState, W = Q + C * LDK, Vt = W + C * kLT, Os = Vt + NV * kLT, kOutput = Os + C * LO;
  static constexpr size_t bytes(bool out, bool bf16) {
    return (size_t)(out ? kOutput : kState) * 4 + (bf16 ? (size_t)C * DK * 2 * (out ? 2 : 1) : 0);
  }
};

template <int DK, int NV, bool kOut>
__global__ void __launch_bounds__(kSimtThreads, DK == 64 ? 2 : 1) chain_simt_kernel(const ChainArgs a) {
  extern __shared__ __align__(16) float sm[];
  using L = ChainSmem<DK, NV>;
  constexpr int LDK = L::LDK, LO = L::LO, JT = NV / 8;
  // P4 tile: DT key rows x JC value columns of both states per thread
  constexpr int DT = (DK == 64 && NV == 8) ? 2 : 4, JC = NV * DK / (kSimtThreads * DT), JG = NV / JC;
  float* St = sm + L::St;      // [2 NV (columns of S, then of M)][LDK (key index)]
  float* Tm = sm + L::T;
  float* Rt = sm + L::Rt;      // R^T
  float4* Wd = reinterpret_cast<float4*>(sm + L::Wd);   // [64][NV] (gS V~, gS V~, gM V~, gM V~): operands of the packed update
  float* Qs = sm + L::Q;
  float* Wm = sm + L::W;
  float* Vt = sm + L::Vt;      // V~^T
  float* Os = sm + L::Os;      // inter-chunk output terms
  uint8_t* raw = reinterpret_cast<uint8_t*>(sm + (kOut ? L::kOutput : L::kState));
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

  auto k_src = [&](const void* p, int c) {
    return static_cast<const void*>(static_cast<const uint8_t*>(p) + ((size_t)(sq.tok0 + c * C) * H + h) * DK * es);
  };
  auto fetch_k = [&](int c) {   // K tile and coefficient vectors of a chunk
    load_rows<DK>(sm + L::K + (c & 1) * C * LDK, raw, k_src(a.k, c), a.in_bf16, (size_t)H * DK, min(C, sq.len - c * C), tid);
    const float* cf = a.coef + ((size_t)(sq.slot0 + c) * H + h) * MDN_NUM_COEF * C;
    if (tid < kChainCoefs * C / 4) cp16(sm + L::cv + (c & 1) * kChainCoefs * C + tid * 4, cf + tid * 4, true);
  };
  auto fetch_q = [&](int c) { load_rows<DK>(Qs, rawQ, k_src(a.q, c), a.in_bf16, (size_t)H * DK, min(C, sq.len - c * C), tid); };
  auto mat = [&](int c) { return ((size_t)(sq.slot0 + c) * H + h) * C * C; };

  if (sq.nchunks > 0) {
    fetch_k(0);
    if (kOut) fetch_q(0);
    load_mat(Tm, a.T + mat(0), tid);
    cp_commit();
  }
  for (int i = tid; i < 2 * NV * DK; i += kSimtThreads) {
    const int jj = i % NV, d = (i / NV) % DK, which = i / (NV * DK);
    const float* src = which ? a.M0 : a.S0;
    St[(which * NV + jj) * LDK + d] = src ? src[st_off + (size_t)d * DV + j0 + jj] : 0.f;
  }

  for (int c = 0; c < sq.nchunks; ++c) {
    const int n = min(C, sq.len - c * C);
    const size_t tok = (size_t)(sq.tok0 + c * C) * H + h;
    const size_t slot_h = (size_t)(sq.slot0 + c) * H + h;
    float* Ks = sm + L::K + (c & 1) * C * LDK;
    const float* cv = sm + L::cv + (c & 1) * kChainCoefs * C;
    cp_wait<0>();
    __syncthreads();   // tiles landed; the previous chunk's readers are done, its state is written
    if (a.in_bf16) {
      widen_tile<DK>(Ks, raw, tid);
      if (kOut) widen_tile<DK>(Qs, rawQ, tid);
      __syncthreads();
    }
    if (c + 1 < sq.nchunks) fetch_k(c + 1);
    if (kOut) load_mat(Wm, a.W + mat(c), tid);
    cp_commit();
    if (!kOut && a.keep_states) {   // the state at the chunk's start, [d][j]
      float* dst = a.keep_states + slot_h * 2 * DK * DV + j0;
      for (int i = tid; i < 2 * NV * DK; i += kSimtThreads) {
        const int j = i % NV, d = (i / NV) % DK, which = i / (NV * DK);
        dst[(size_t)which * DK * DV + (size_t)d * DV + j] = St[(which * NV + j) * LDK + d];
      }
    }

    // ---- 1: K S, K M (row slots 0..15), Q S, Q M (16..31): rows slot + 16 i, columns jg + 8 jj of both states
    // (without the output terms: K S, K M on all slots, rows slot + 32 i)
    {
      constexpr int RT = kOut ? 4 : 2, RS = C / RT;
      const bool q_rows = kOut && rs >= RS;
      const int r0 = rs & (RS - 1);
      float vv[RT][JT];
      if (!q_rows) {
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
          for (int jj = 0; jj < JT; ++jj)
            vv[i][jj] = r0 + RS * i < n ? load_io(a.v, (tok + (size_t)(r0 + RS * i) * H) * DV + j0 + jg + 8 * jj, a.in_bf16) : 0.f;
      }
      float2 acc[RT][2 * JT];
      zero2(acc);
      dot_tile<RT, 2 * JT>(acc, (q_rows ? Qs : Ks) + r0 * LDK, RS * LDK, St + jg * LDK, 8 * LDK, 0, DK / 4);
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const int r = r0 + RS * i;
        const float ab = cv[kAbar * C + r], w = cv[(q_rows ? kB : kAlphaBPrev) * C + r];
#pragma unroll
        for (int jj = 0; jj < JT; ++jj) {
          const float xs = hsum(acc[i][jj]), xm = hsum(acc[i][JT + jj]);
          if (!q_rows) Rt[(jg + 8 * jj) * kLT + r] = vv[i][jj] - ab * xs + w * xm;
          else Os[r * LO + jg + 8 * jj] = a.scale * (ab * xs - w * xm);
        }
      }
    }
    __syncthreads();
    if (kOut && c + 1 < sq.nchunks) fetch_q(c + 1);   // Q has been read
    cp_commit();

    // ---- 2: V~ = T R (T lower triangular): rows rs, rs + 32
    {
      float2 acc[2][JT];
      zero2(acc);
      dot_tile<2, JT>(acc, Tm + rs * kLT, 32 * kLT, Rt + jg * kLT, 8 * kLT, 0, 8);
      float2 hi[1][JT];
#pragma unroll
      for (int jj = 0; jj < JT; ++jj) hi[0][jj] = acc[1][jj];
      dot_tile<1, JT>(hi, Tm + (rs + 32) * kLT, 0, Rt + jg * kLT, 8 * kLT, 8, 16);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = rs + 32 * i;
        const float gs = cv[kGS * C + r], gm = cv[kGM * C + r];
#pragma unroll
        for (int jj = 0; jj < JT; ++jj) {
          const float x = i ? hsum(hi[0][jj]) : hsum(acc[0][jj]);
          const int j = jg + 8 * jj;
          if (kOut) Vt[j * kLT + r] = x;
          else a.keep_vt[(slot_h * C + r) * DV + j0 + j] = x;
          Wd[r * NV + j] = make_float4(gs * x, gs * x, gm * x, gm * x);
        }
      }
    }
    if (kOut) cp_wait<1>();   // W is in (the next Q may be on its way)
    __syncthreads();
    if (c + 1 < sq.nchunks) load_mat(Tm, a.T + mat(c + 1), tid);   // T has been read
    cp_commit();

    // ---- 3: O = inter + W V~
    if (kOut) {
      float2 acc[2][JT];
      zero2(acc);
      dot_tile<2, JT>(acc, Wm + rs * kLT, 32 * kLT, Vt + jg * kLT, 8 * kLT, 0, 8);
      float2 hi[1][JT];
#pragma unroll
      for (int jj = 0; jj < JT; ++jj) hi[0][jj] = acc[1][jj];
      dot_tile<1, JT>(hi, Wm + (rs + 32) * kLT, 0, Vt + jg * kLT, 8 * kLT, 8, 16);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = rs + 32 * i;
#pragma unroll
        for (int jj = 0; jj < JT; ++jj) {
          const int j = jg + 8 * jj;
          if (r < n) store_io(a.o, (tok + (size_t)r * H) * DV + j0 + j, a.o_bf16, Os[r * LO + j] + (i ? hsum(hi[0][jj]) : hsum(acc[0][jj])));
        }
      }
    }

    // ---- 4: state hand-over, DT key rows x JC columns of S and M per thread (each entry has one owner: no barrier)
    {
      const int lane = tid & 31, warp = tid >> 5;
      constexpr int DB = DK / DT / 8;   // key-row blocks of eight groups
      const int d0 = ((warp % DB) * 8 + (lane & 7)) * DT, jq = (warp / DB) * 4 + (lane >> 3);
      float2 acc[2 * JC][DT / 2];
      zero2(acc);
      const float* kp = Ks + d0;
      const float4* wp = Wd + jq;
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
      const float aC = cv[kAbar * C + C - 1], bC = cv[kB * C + C - 1], mC = cv[kMubar * C + C - 1];
#pragma unroll
      for (int jc = 0; jc < JC; ++jc) {
        float* sp = St + (jq + JG * jc) * LDK + d0;
        float* mp = sp + NV * LDK;
#pragma unroll
        for (int p = 0; p < DT / 2; ++p) {
          const float2 s = *reinterpret_cast<float2*>(sp + 2 * p), m = *reinterpret_cast<float2*>(mp + 2 * p);
          const float2 ds = acc[2 * jc][p], dm = acc[2 * jc + 1][p];
          *reinterpret_cast<float2*>(sp + 2 * p) = make_float2(aC * s.x - bC * m.x + ds.x, aC * s.y - bC * m.y + ds.y);
          *reinterpret_cast<float2*>(mp + 2 * p) = make_float2(mC * m.x - dm.x, mC * m.y - dm.y);
        }
      }
    }
  }
  cp_wait<0>();
  __syncthreads();
  for (int i = tid; i < 2 * NV * DK; i += kSimtThreads) {
    const int jj = i % NV, d = (i / NV) % DK, which = i / (NV * DK);
    float* dst = which ? a.Mf : a.Sf;
    if (dst) dst[st_off + (size_t)d * DV + j0 + jj] = St[(which * NV + jj) * LDK + d];
  }
}

template <int DK, int NV, bool kOut> cudaError_t launch_one(const Plan& pl, const ChainArgs& a) {
  const size_t smem = ChainSmem<DK, NV>::bytes(kOut, a.in_bf16);
  auto kern = chain_simt_kernel<DK, NV, kOut>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)pl.geom.num_seqs * pl.p.H * (a.dv / NV);
  return launch_pdl(kern, dim3(grid), dim3(kSimtThreads), smem, pl.stream, a);
}

template <bool kOut> cudaError_t launch_dims(const Plan& pl, const ChainArgs& a) {
  const bool narrow = simt_narrow_columns(pl);
  if (pl.p.dk == 64) return narrow ? launch_one<64, 8, kOut>(pl, a) : launch_one<64, 16, kOut>(pl, a);
  return narrow ? launch_one<128, 8, kOut>(pl, a) : launch_one<128, 16, kOut>(pl, a);
}

ChainArgs chain_args(const Plan& pl, const void* q, const void* k, const void* v, const float* S0, const float* M0) {
  ChainArgs a{};
  a.g = pl.geom;
  a.q = q; a.k = k; a.v = v;
  a.in_bf16 = pl.p.io_dtype == MDN_BF16; a.o_bf16 = pl.p.o_dtype == MDN_BF16;
  a.dv = pl.p.dv;
  a.coef = reinterpret_cast<const float*>(pl.ws + pl.lay.off_coef);
  a.T = reinterpret_cast<const float*>(pl.ws + pl.lay.off_T);
  a.W = reinterpret_cast<const float*>(pl.ws + pl.lay.off_W);
  a.S0 = S0; a.M0 = M0;
  a.scale = pl.p.scale;
  return a;
}

}  // namespace

// Eight value columns per CTA as long as that makes no more CTAs than SMs (a chunk's latency is what counts then);
// sixteen beyond (twice the arithmetic per operand load).
bool simt_narrow_columns(const Plan& pl) { return (int64_t)pl.geom.num_seqs * pl.p.H * (pl.p.dv / 8) <= 148; }

cudaError_t launch_chain_simt(const Plan& pl, const void* q, const void* k, const void* v, const float* S0,
                              const float* M0, void* o, float* Sf, float* Mf, int* launches) {
  ChainArgs a = chain_args(pl, q, k, v, S0, M0);
  a.o = o; a.Sf = Sf; a.Mf = Mf;
  const cudaError_t e = launch_dims<true>(pl, a);
  if (e == cudaSuccess) ++*launches;
  return e;
}

cudaError_t launch_chain_simt_keep(const Plan& pl, const void* k, const void* v, const float* S0, const float* M0,
                                   float* states, float* vt, int* launches) {
  ChainArgs a = chain_args(pl, nullptr, k, v, S0, M0);
  a.keep_states = states; a.keep_vt = vt;
  const cudaError_t e = launch_dims<false>(pl, a);
  if (e == cudaSuccess) ++*launches;
  return e;
}

}  // namespace mdn
