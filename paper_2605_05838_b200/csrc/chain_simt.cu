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
// What bounds it: the chunks are serial, so a chunk's latency is the kernel's time: four products (five with the output)
// between three barriers, each bound by the shared-memory port (simt_tile.cuh: 8 x 8 tiles per thread with the summed
// index split over lanes, because a chunk has only 32 to 64 such tiles of outputs).  Hence NV is small (8 columns while
// that makes no more CTAs than SMs, else 16), and the next chunk's K, Q, T, W are fetched by cp.async into buffers as they
// fall free (K twice buffered: it is the first and the last operand of a chunk).
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
  int short_limit;      // kOut = false: sequences of up to so many tokens are left out
};

template <int DK, int NV> struct ChainSmem {   // float offsets
  static constexpr int LDK = DK + 4, LO = NV == 8 ? 8 : NV + 8;
  static constexpr int K = 0, St = K + 2 * C * LDK, T = St + 2 * NV * LDK, Rt = T + C * kLT, Wd = Rt + NV * kLT,
                       cv = Wd + C * (2 * NV + 4), kState = cv + 2 * kChainCoefs * C;
  static constexpr int Q = kState, W = Q + C * LDK, Vt = W + C * kLT, Os = Vt + NV * kLT, kOutput = Os + C * LO;
  static constexpr size_t bytes(bool out, bool bf16) {
    return (size_t)(out ? kOutput : kState) * 4 + (bf16 ? (size_t)C * DK * 2 * (out ? 2 : 1) : 0);
  }
};

template <int DK, int NV, bool kOut>
__global__ void __launch_bounds__(kChainThreads<NV>, 1) chain_simt_kernel(const ChainArgs a) {
  extern __shared__ __align__(16) float sm[];
  using L = ChainSmem<DK, NV>;
  constexpr int TH = kChainThreads<NV>, LDK = L::LDK, LO = L::LO, LDW = 2 * NV + 4;
  float* St = sm + L::St;      // [2 NV (columns of S, then of M)][LDK (key index)]
  float* Tm = sm + L::T;
  float* Rt = sm + L::Rt;      // R^T
  float* Wd = sm + L::Wd;      // [64][LDW]: (gS V~, gM V~) per column, the weights of the state update
  float* Qs = sm + L::Q;
  float* Wm = sm + L::W;
  float* Vt = sm + L::Vt;      // V~^T
  float* Os = sm + L::Os;      // inter-chunk output terms
  uint8_t* raw = reinterpret_cast<uint8_t*>(sm + (kOut ? L::kOutput : L::kState));
  uint8_t* rawQ = raw + C * DK * 2;

  const int tid = threadIdx.x;
  const StateTile<NV, kOut ? 2 : 1> st_tile(tid);
  const TriTile<NV> tri(tid);
  const int H = a.g.H, DV = a.dv, NVB = DV / NV;
  const int vb = blockIdx.x % NVB, h = (blockIdx.x / NVB) % H, seq = blockIdx.x / (NVB * H);
  const int j0 = vb * NV;
  grid_dependency_wait();
  grid_launch_dependents();
  const SeqInfo sq = seq_info(a.g, seq);
  if (!kOut && short_sequence(sq, a.short_limit)) return;
  const size_t st_off = ((size_t)seq * H + h) * DK * DV;
  const size_t es = a.in_bf16 ? 2 : 4;

  auto k_src = [&](const void* p, int c) {
    return static_cast<const void*>(static_cast<const uint8_t*>(p) + ((size_t)(sq.tok0 + c * C) * H + h) * DK * es);
  };
  auto fetch_k = [&](int c) {   // K tile and coefficient vectors of a chunk
    load_rows<DK, TH>(sm + L::K + (c & 1) * C * LDK, raw, k_src(a.k, c), a.in_bf16, (size_t)H * DK, min(C, sq.len - c * C), tid);
    const float* cf = a.coef + ((size_t)(sq.slot0 + c) * H + h) * MDN_NUM_COEF * C;
    if (tid < kChainCoefs * C / 4) cp16(sm + L::cv + (c & 1) * kChainCoefs * C + tid * 4, cf + tid * 4, true);
  };
  auto fetch_q = [&](int c) { load_rows<DK, TH>(Qs, rawQ, k_src(a.q, c), a.in_bf16, (size_t)H * DK, min(C, sq.len - c * C), tid); };
  auto mat = [&](int c) { return ((size_t)(sq.slot0 + c) * H + h) * C * C; };

  if (sq.nchunks > 0) {
    fetch_k(0);
    if (kOut) fetch_q(0);
    load_mat<TH>(Tm, a.T + mat(0), tid);
    cp_commit();
  }
  for (int i = tid; i < 2 * NV * DK; i += TH) {
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
      widen_tile<DK, TH>(Ks, raw, tid);
      if (kOut) widen_tile<DK, TH>(Qs, rawQ, tid);
      __syncthreads();
    }
    if (c + 1 < sq.nchunks) fetch_k(c + 1);
    if (kOut) load_mat<TH>(Wm, a.W + mat(c), tid);
    cp_commit();
    if (!kOut && a.keep_states) {   // the state at the chunk's start, [d][j]
      float* dst = a.keep_states + slot_h * 2 * DK * DV + j0;
      for (int i = tid; i < 2 * NV * DK; i += TH) {
        const int j = i % NV, d = (i / NV) % DK, which = i / (NV * DK);
        dst[(size_t)which * DK * DV + (size_t)d * DV + j] = St[(which * NV + j) * LDK + d];
      }
    }

    // ---- 1: K S, K M -> R;  Q S, Q M -> the inter-chunk output terms
    {
      float vv[st_tile.kPairs];
      st_tile.own([&](int e, int which, int r, int j) {
        vv[e] = which == 0 && r < n ? load_io(a.v, (tok + (size_t)r * H) * DV + j0 + j, a.in_bf16) : 0.f;
      });
      st_tile.template run<DK>(Ks, Qs, St, [&](int e, int which, int r, int j, float xs, float xm) {
        const float ab = cv[kAbar * C + r];
        if (which == 0) Rt[j * kLT + r] = vv[e] - ab * xs + cv[kAlphaBPrev * C + r] * xm;
        else Os[r * LO + j] = a.scale * (ab * xs - cv[kB * C + r] * xm);
      });
    }
    __syncthreads();
    if (kOut && c + 1 < sq.nchunks) fetch_q(c + 1);   // Q has been read
    cp_commit();

    // ---- 2: V~ = T R  (T lower triangular)
    tri.template run<true>(Tm, Rt, [&](int r, int j, float x) {
      if (kOut) Vt[j * kLT + r] = x;
      else a.keep_vt[(slot_h * C + r) * DV + j0 + j] = x;
      *reinterpret_cast<float2*>(Wd + r * LDW + 2 * j) = make_float2(cv[kGS * C + r] * x, cv[kGM * C + r] * x);
    });
    if (kOut) cp_wait<1>();   // W is in (the next Q may be on its way)
    __syncthreads();
    if (c + 1 < sq.nchunks) load_mat<TH>(Tm, a.T + mat(c + 1), tid);   // T has been read
    cp_commit();

    // ---- 3: O = inter + W V~
    if (kOut)
      tri.template run<true>(Wm, Vt, [&](int r, int j, float x) {
        if (r < n) store_io(a.o, (tok + (size_t)r * H) * DV + j0 + j, a.o_bf16, Os[r * LO + j] + x);
      });

    // ---- 4: state hand-over (each entry has one owner: no barrier)
    {
      UpdateTile<DK, NV> up(tid);
      up.add(Ks, Wd, n);
      const float aC = cv[kAbar * C + C - 1], bC = cv[kB * C + C - 1], mC = cv[kMubar * C + C - 1];
      up.finish([&](int d, int j, float ds, float dm) {
        float* sp = St + j * LDK + d;
        float* mp = sp + NV * LDK;
        const float s = *sp, m = *mp;
        *sp = aC * s - bC * m + ds;
        *mp = mC * m - dm;
      });
    }
  }
  cp_wait<0>();
  __syncthreads();
  for (int i = tid; i < 2 * NV * DK; i += TH) {
    const int jj = i % NV, d = (i / NV) % DK, which = i / (NV * DK);
    float* dst = which ? a.Mf : a.Sf;
    if (dst) dst[st_off + (size_t)d * DV + j0 + jj] = St[(which * NV + jj) * LDK + d];
  }
}

template <int DK, int NV, bool kOut> cudaError_t launch_one(const Plan& pl, const ChainArgs& a) {
  const size_t smem = ChainSmem<DK, NV>::bytes(kOut, a.in_bf16);
  auto kern = chain_simt_kernel<DK, NV, kOut>;
  const cudaError_t e = allow_smem<(int)ChainSmem<DK, NV>::bytes(kOut, true)>(kern);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)pl.geom.num_seqs * pl.p.H * (a.dv / NV);
  return launch_pdl(kern, dim3(grid), dim3(kChainThreads<NV>), smem, pl.stream, a);
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
bool simt_narrow_columns(const Plan& pl) { return (int64_t)pl.geom.num_seqs * pl.p.H * (pl.p.dv / 8) <= kSms; }

cudaError_t launch_chain_simt(const Plan& pl, const void* q, const void* k, const void* v, const float* S0,
                              const float* M0, void* o, float* Sf, float* Mf, int* launches) {
  ChainArgs a = chain_args(pl, q, k, v, S0, M0);
  a.o = o; a.Sf = Sf; a.Mf = Mf;
  const cudaError_t e = launch_dims<true>(pl, a);
  if (e == cudaSuccess) ++*launches;
  return e;
}

cudaError_t launch_chain_simt_keep(const Plan& pl, const void* k, const void* v, const float* S0, const float* M0,
                                   float* states, float* vt, int short_limit, int* launches) {
  ChainArgs a = chain_args(pl, nullptr, k, v, S0, M0);
  a.keep_states = states; a.keep_vt = vt;
  a.short_limit = short_limit;
  const cudaError_t e = launch_dims<false>(pl, a);
  if (e == cudaSuccess) ++*launches;
  return e;
}

}  // namespace mdn
