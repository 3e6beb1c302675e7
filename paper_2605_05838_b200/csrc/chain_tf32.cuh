// What the two chain kernels on tf32 state operands share (chain_tf32.cu: one CTA per chain; chain_half.cu: one CTA per half of a
// chain's value columns): arguments, which run a CTA makes, and the per-chunk coefficients of the lazily scaled state.
#pragma once

#include "mdn_common.cuh"

namespace mdn {

// per-chunk block the producer warp publishes (float indices)
enum Adj : int { kCx = 0, kCy = 64, kCz = 128, kCu = 192, kWs = 256, kWm = 320, kN11 = 384, kN12, kN22, kLazy };
constexpr uint32_t kAdjBytes = 2048;
constexpr float kLazyMin = 5.421010862427522e-20f;   // 2^-64: smallest g11', g22' a lazy chunk may leave
constexpr float kLazyMix = 1.f;                      // largest |g12'| / g22' (beyond it the two hat terms of S cancel too much)

// Debug builds: the chunks that are stamped.  The buffer holds 24 rows of 32 words; the words before the first stamped chunk's row
// take the run's own stamps.
constexpr int kTlFirst = 16, kTlChunks = 8;
static_assert((kTlFirst + kTlChunks) * 32 <= 24 * 32, "the documented size of the buffer");

struct ChainTf32Args {
  ChunkGeom g;
  const float* coef;
  const float* S0;
  const float* M0;
  void* o;
  float* Sf;
  float* Mf;
  int32_t* status;
  float scale;
  // parallel inter-chunk scan (seg_G = 0: off, one run walks all chunks of its chain)
  int seg_G;
  int seg_phase;
  int seg_first, seg_mid, seg_least;   // see seg_chunks
  float* seg_E;
  float* seg_Psi;
  float* seg_PhiS;
  float* seg_PhiM;
  long long* timeline;   // debug builds: CTA 0 writes clock64() at [chunk * 32 + event], chunks kTlFirst .. kTlFirst + 7
  // layer operations (Section 3.3), kLayer instantiation only
  int qk_on;             // q <- L2Norm(q - d k), k <- L2Norm(k): 1/|k|, 1/|q - d k| arrive as coefficient vectors 6, 7
  const float* qk_d;     // [H] or NULL
  int post_on;           // o <- sigmoid(g) * RMSNorm(o) * w in the output step
  const float* post_w;   // [dv] or NULL
  const void* post_g;    // [B,T,H,dv] bf16
  float post_eps;
};

__device__ __forceinline__ float sigmoid_fast(float x) {
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(0.5f * x));
  return fmaf(0.5f, t, 0.5f);
}

// One run over consecutive chunks of a chain: which chunks, where the start state comes from (NULL: zero, or the identity in the
// half that id_s / id_m names), where the end state goes, whether V counts and o is written.
struct ChainRun {
  SeqInfo sq;
  int h;
  const float* S0;
  const float* M0;
  float* Sf;
  float* Mf;
  bool id_s, id_m, v_zero, write_o;
};
__device__ __forceinline__ ChainRun chain_run(const ChainTf32Args& a, int item) {
  constexpr int kD = 128;
  constexpr size_t kMat = (size_t)kD * kD;
  const int H = a.g.H;
  int chain = item, seg = 0, run = 0;   // run 0: the real thing; 1: Psi; 2: Phi from (I, 0); 3: Phi from (0, I)
  if (a.seg_G > 0) {
    if (a.seg_phase == 1) {   // the first segments (the longest runs) lead
      const int chains = a.g.num_seqs * H, items = 3 * (a.seg_G - 2), w = item - chains;
      if (w >= 0) {
        chain = w / items;
        seg = 1 + (w % items) / 3;
        run = 1 + (w % items) % 3;
      }
    } else {
      chain = item / (a.seg_G - 1);
      seg = 1 + item % (a.seg_G - 1);
    }
  }
  const int seq = chain / H;
  ChainRun r;
  r.h = chain % H;
  r.sq = seq_info(a.g, seq);
  if (a.seg_G > 0) {        // restrict the view to this segment's chunks
    const int2 span = seg_chunks(a.g, r.sq.nchunks, SegSplitArgs{a.seg_G, a.seg_first, a.seg_mid, a.seg_least}, seg);
    const int cb = span.x, ce = span.y;
    r.sq.slot0 += cb;
    r.sq.tok0 += cb * C;
    r.sq.len = (ce > cb) ? min(r.sq.len - cb * C, (ce - cb) * C) : 0;
    r.sq.nchunks = ce - cb;
  }
  const size_t st_off = (size_t)chain * kMat;
  r.S0 = a.S0 ? a.S0 + st_off : nullptr;
  r.M0 = a.M0 ? a.M0 + st_off : nullptr;
  r.Sf = a.Sf ? a.Sf + st_off : nullptr;
  r.Mf = a.Mf ? a.Mf + st_off : nullptr;
  r.id_s = r.id_m = r.v_zero = false;
  r.write_o = true;
  if (a.seg_G > 0) {
    auto e_ptr = [&](int gi, int which) { return a.seg_E + (((size_t)chain * (a.seg_G - 1) + gi) * 2 + which) * kMat; };
    if (run == 0) {
      if (seg > 0) { r.S0 = e_ptr(seg - 1, 0); r.M0 = e_ptr(seg - 1, 1); }
      if (seg < a.seg_G - 1) {
        r.Sf = (seg == 0) ? e_ptr(0, 0) : nullptr;
        r.Mf = (seg == 0) ? e_ptr(0, 1) : nullptr;
      }
    } else {
      r.write_o = false;
      r.S0 = r.M0 = nullptr;
      r.id_s = run == 2; r.id_m = run == 3; r.v_zero = run >= 2;
      float* base = (run == 1 ? a.seg_Psi : run == 2 ? a.seg_PhiS : a.seg_PhiM) +
                    (((size_t)chain * (a.seg_G - 2) + (seg - 1)) * 2) * kMat;
      r.Sf = base; r.Mf = base + kMat;
    }
  }
  return r;
}

// The scalar recurrence of G = [[g11, g12], [0, g22]] over one chunk and the chunk's six coefficient vectors (two tokens per lane
// of the calling warp), from its coefficient vectors cf to the published block aj.
template <bool kLayer>
__device__ __forceinline__ void publish_coefs(const float* cf, float* aj, float scale, int lane, float& g11, float& g12, float& g22) {
  const float aC = cf[kAbar * C + C - 1], bC = cf[kB * C + C - 1], mC = cf[kMubar * C + C - 1];
  const float n11 = __fmul_rn(aC, g11), n12 = __fsub_rn(__fmul_rn(aC, g12), __fmul_rn(bC, g22)), n22 = __fmul_rn(mC, g22);
  const bool lazy = n11 >= kLazyMin && n22 >= kLazyMin && fabsf(n12) <= kLazyMix * n22;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int t = 2 * lane + e;
    const float ab = cf[kAbar * C + t], bb = cf[kB * C + t], pp = cf[kAlphaBPrev * C + t];
    const float gs = cf[kGS * C + t], gm = cf[kGM * C + t];
    // fused q/k norm: k^ = k / |k| scales the rows of K S, K M (vectors 2, 3, 4 carry that factor already),
    // q^ = (q - d k) / |q - d k| those of the output terms (the converter warps subtract d k from the Q tile)
    float cx, cy, cz, cu;
    if constexpr (kLayer) {
      const float rk = cf[kRk * C + t], sq_ = scale * cf[kRq * C + t];
      cx = ab * rk * g11; cy = pp * g22 - ab * rk * g12;
      cz = sq_ * (ab * g11); cu = sq_ * (ab * g12 - bb * g22);
    } else {
      cx = ab * g11; cy = pp * g22 - ab * g12;
      cz = scale * cx; cu = scale * (ab * g12 - bb * g22);
    }
    aj[kCx + t] = -cx;     // stored negated: the epilogue's first step is one packed FMA per token pair
    aj[kCy + t] = cy;
    aj[kCz + t] = cz;
    aj[kCu + t] = cu;
    aj[kWs + t] = lazy ? (gs + (n12 / n22) * gm) / n11 : gs;
    aj[kWm + t] = lazy ? gm / n22 : gm;
  }
  if (lane == 0) { aj[kN11] = n11; aj[kN12] = n12; aj[kN22] = n22; aj[kLazy] = lazy ? 1.f : 0.f; }
  if (lazy) { g11 = n11; g12 = n12; g22 = n22; } else { g11 = 1.f; g12 = 0.f; g22 = 1.f; }
}

// S = g11 Sh + g12 Mh, one element: of the masters that an eager chunk rescales, and of a final state.
__device__ __forceinline__ float unscale_s(float g11, float s, float g12, float m) { return fmaf(g11, s, __fmul_rn(g12, m)); }
__device__ __forceinline__ float final_s(float g11, float s, float g12, float m) { return fmaf(g12, m, __fmul_rn(g11, s)); }

// chain_half.cu: `items` runs (of a launch described by a), two CTAs each.
struct ChainTensors { const void* q; const void* k; const void* v; };
cudaError_t launch_chain_half(const Plan& pl, const ChainTf32Args& a, const ChainTensors& in, unsigned items, int* launches);

}  // namespace mdn
