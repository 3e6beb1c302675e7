// a1 + a2 in fp32: per (chunk, head) the coefficient scan of Eq. 10, the intra-chunk system of Eq. 15 and the masked
// query-key matrix of Eq. 12.
//
//   gamma_{r,i} = alpha_r gamma_{r-1,i} + beta_r m_{r,i},  m_{r,i} = mu_r m_{r-1,i}, m_{i,i} = 1     (thread = column i)
//   A[r][i]     = alpha_r gamma_{r-1,i} eta_i (k_r . k_i)       (i < r)    = ((P K^T) .* Gamma^-)[r][i]
//   T           = (I + A)^{-1}             blocked: 16 x 16 diagonal blocks by forward substitution, then
//                                          T_21 = -T_22 A_21 T_11 at block sizes 16 and 32
//   W[r][i]     = scale gamma_{r,i} eta_i (q_r . k_i)           (i <= r)
//
// Gamma^- is Gamma shifted down one row (the derivation substitutes S_{t-1}); with
// p_r = alpha_r k_r its entry is alpha_r gamma_{r-1,i}, which the column recurrence
// produces directly, with no subtraction.  All arithmetic fp32; q, k are widened on load.
//
// One 256-thread CTA per (chunk, head).  What bounds it at few chunks is its own latency: the scan and the recurrence
// of gamma run on three warps while K and Q are on their way, [K; Q] K^T is one register-tiled product that skips the
// 8 x 16 blocks above the diagonal, and the inverse is seven short parallel steps instead of 64 dependent rows.
// Two CTAs per SM (93 KB at dk = 128): A, W and T live where K, Q and Gamma were.
#include <type_traits>

#include "coeff_scan.cuh"
#include "simt_tile.cuh"

namespace mdn {
namespace {

struct IntraArgs {
  ChunkGeom g;
  const void* q; const void* k;
  bool in_bf16;
  float* coef;
  GateArgs gates;
  GateParam gp;
  float scale;
  float* T; float* W;
  IntraBwd bwd;           // set for the exact backward: T, T^T and W^T dO leave instead of T and W
  int dv;
  bool do_bf16;
  int32_t* clear_status;  // or NULL: the status word, when this is the call's first kernel
};

template <int DK> struct IntraSmem {   // float offsets
  static constexpr int LDK = DK + 4, K = 0, Q = K + C * LDK, G = Q + C * LDK, P = G + C * kLT, cv = P + 32 * 36, kFloats = cv + 4 * C;
  static constexpr size_t bytes(bool bf16, int dv_bwd) {   // dv_bwd: dv for the exact backward (the dO tile), else 0
    return (size_t)kFloats * 4 + (bf16 ? (size_t)2 * C * DK * 2 : 0) + (dv_bwd ? (size_t)C * (dv_bwd + 4) * 4 : 0);
  }
};

template <int DK>
__global__ void __launch_bounds__(kSimtThreads, 2) intra_simt_kernel(const IntraArgs a) {
  extern __shared__ __align__(16) float sm[];
  using L = IntraSmem<DK>;
  constexpr int LDK = L::LDK, LP = 36;
  const int H = a.g.H, slot = blockIdx.x / H, h = blockIdx.x % H;
  grid_dependency_wait();
  grid_launch_dependents();
  if (a.clear_status != nullptr && blockIdx.x == 0 && threadIdx.x < 4) a.clear_status[threadIdx.x] = 0;
  const SlotInfo si = slot_info(a.g, slot);
  if (si.seq < 0 || (a.bwd.TT != nullptr && short_sequence(si, a.bwd.short_limit))) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* Ks = sm + L::K;
  float* Qs = sm + L::Q;
  float* Gs = sm + L::G;       // gamma; then T
  float* Ps = sm + L::P;       // scratch of the inverse
  float* cv = sm + L::cv;      // alpha, beta, mu, eta
  float* As = Ks;              // after the product: A, W in the place of K, Q
  float* Ws = Qs;
  float* Ts = Gs;
  uint8_t* raw = reinterpret_cast<uint8_t*>(sm + L::kFloats);

  const size_t es = a.in_bf16 ? 2 : 4, row0 = ((size_t)si.tok0 * H + h) * DK * es;
  load_rows<DK>(Ks, raw, static_cast<const uint8_t*>(a.k) + row0, a.in_bf16, (size_t)H * DK, si.n, tid);
  load_rows<DK>(Qs, raw + C * DK * 2, static_cast<const uint8_t*>(a.q) + row0, a.in_bf16, (size_t)H * DK, si.n, tid);
  const int LDV = a.dv + 4;
  float* Do = reinterpret_cast<float*>(raw + (a.in_bf16 ? 2 * C * DK * 2 : 0));
  if (a.bwd.TT != nullptr)
    load_io_rows(Do, static_cast<const uint8_t*>(a.bwd.d_o) + ((size_t)si.tok0 * H + h) * a.dv * (a.do_bf16 ? 2 : 4), a.do_bf16, a.dv,
                 (size_t)H * a.dv, si.n, tid);
  cp_commit();

  float* cf = a.coef + ((size_t)slot * H + h) * MDN_NUM_COEF * C;
  if (a.gates.log_alpha == nullptr) {   // the scan has run: its gate vectors are in the workspace
    cv[tid] = cf[kAlpha * C + tid];
    __syncthreads();
  } else {
    if (tid < C) {
      TokenGates tg{1.f, 1.f, 0.f, 0.f};   // exact no-ops past the end of a short chunk
      if (tid < si.n) {
        const size_t gi = ((size_t)si.tok0 + tid) * H + h;
        tg = load_token_gates(a.gp, h, __ldg(a.gates.log_alpha + gi), __ldg(a.gates.log_mu + gi), __ldg(a.gates.beta + gi),
                              a.gates.eta ? __ldg(a.gates.eta + gi) : 1.f);
      }
      cv[0 * C + tid] = tg.alpha; cv[1 * C + tid] = tg.beta; cv[2 * C + tid] = tg.mu; cv[3 * C + tid] = tg.eta;
    }
    __syncthreads();
    if (warp == 2) {
      const float2 a2 = reinterpret_cast<const float2*>(cv)[lane], b2 = reinterpret_cast<const float2*>(cv + C)[lane];
      const float2 m2 = reinterpret_cast<const float2*>(cv + 2 * C)[lane], e2 = reinterpret_cast<const float2*>(cv + 3 * C)[lane];
      const float al[2] = {a2.x, a2.y}, be[2] = {b2.x, b2.y}, mu[2] = {m2.x, m2.y}, et[2] = {e2.x, e2.y};
      const HeadCoefs hc = scan_head(al, mu, be, et, lane);
      auto put = [&](int which, float x0, float x1) { reinterpret_cast<float2*>(cf + which * C)[lane] = make_float2(x0, x1); };
      put(kAbar, hc.abar[0], hc.abar[1]);
      put(kB, hc.b[0], hc.b[1]);
      put(kAlphaBPrev, hc.ab_prev[0], hc.ab_prev[1]);
      put(kGS, hc.gs[0], hc.gs[1]);
      put(kGM, hc.gm[0], hc.gm[1]);
      put(kMubar, hc.mubar[0], hc.mubar[1]);
      put(kRk, 1.f, 1.f);
      put(kRq, 1.f, 1.f);
      put(kAlpha, al[0], al[1]);
      put(kBeta, be[0], be[1]);
      put(kMu, mu[0], mu[1]);
      put(kEta, et[0], et[1]);
    }
  }
  if (tid < C) {   // column i of Gamma (zero above the diagonal)
    const int i = tid;
    float m = 1.f, gam = 0.f;
#pragma unroll 4
    for (int rb = 0; rb < C; rb += 4) {
      const float4 al = lds4(cv + rb), be = lds4(cv + C + rb), mu = lds4(cv + 2 * C + rb);
      const float a4[4] = {al.x, al.y, al.z, al.w}, b4[4] = {be.x, be.y, be.z, be.w}, m4[4] = {mu.x, mu.y, mu.z, mu.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = rb + u;
        if (r > i) m *= m4[u];
        if (r >= i) gam = fmaf(a4[u], gam, b4[u] * m);
        Gs[r * kLT + i] = r >= i ? gam : 0.f;
      }
    }
  }
  cp_wait<0>();
  __syncthreads();
  if (a.in_bf16) {
    widen_tile<DK>(Ks, raw, tid);
    widen_tile<DK>(Qs, raw + C * DK * 2, tid);
    __syncthreads();
  }

  // ---- [K; Q] K^T: rows r0 + 16 i (row slots 0..15: K, 16..31: Q), columns jg + 8 jj; block i reaches columns 16 i + 15
  const int jg = tid & 7, rs = tid >> 3, r0 = rs & 15;
  const bool w_rows = rs >= 16;
  float out[4][8];
  {
    float2 acc[4][8];
    zero2(acc);
    const float* ap = (w_rows ? Qs : Ks) + r0 * LDK;
    const float* bp = Ks + jg * LDK;
#pragma unroll 1
    for (int k = 0; k < DK; k += 4) {
      float4 av[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = lds4(ap + i * 16 * LDK + k);
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const float4 bv = lds4(bp + jj * 8 * LDK + k);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (jj <= 2 * i + 1) fma4(acc[i][jj], av[i], bv);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) out[i][jj] = hsum(acc[i][jj]);
  }
  __syncthreads();   // K and Q have been read
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + 16 * i;
    const float f = w_rows ? a.scale : cv[r];
    const float* grow = Gs + (w_rows ? r : max(r - 1, 0)) * kLT;
    float* dst = (w_rows ? Ws : As) + r * kLT;
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) {
      const int c = jg + 8 * jj;
      const bool in = w_rows ? c <= r : c < r;
      dst[c] = in ? f * grow[c] * cv[3 * C + c] * out[i][jj] : 0.f;
    }
  }
  __syncthreads();   // A, W complete; Gamma has been read: T takes its place

  const size_t mat = ((size_t)slot * H + h) * C * C;
  if (a.bwd.TT != nullptr) {   // W^T dO: eight rows per warp (W read as it lies: its row r is the update by dO's row r)
    const int i0 = warp * 8;
    float* dst = a.bwd.vp + (((size_t)slot * H + h) * C + i0) * a.dv;
    auto columns = [&](auto width) {
      constexpr int W2 = decltype(width)::value;   // float2 column pairs per lane
      float2 acc[8][W2];
      zero2(acc);
#pragma unroll 2
      for (int r = i0; r < si.n; ++r) {
        const float4 wa = lds4(Ws + r * kLT + i0), wb = lds4(Ws + r * kLT + i0 + 4);
        const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
        float2 d[W2];
#pragma unroll
        for (int e = 0; e < W2; ++e) d[e] = *reinterpret_cast<const float2*>(Do + r * LDV + 2 * lane + 64 * e);
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int e = 0; e < W2; ++e) acc[i][e] = __ffma2_rn(make_float2(w[i], w[i]), d[e], acc[i][e]);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int e = 0; e < W2; ++e) *reinterpret_cast<float2*>(dst + (size_t)i * a.dv + 2 * lane + 64 * e) = acc[i][e];
    };
    if (a.dv == 64) columns(std::integral_constant<int, 1>{});
    else columns(std::integral_constant<int, 2>{});
  }
  // step 1: the four diagonal blocks (thread = block, column); the other threads clear the blocks above the diagonal and
  // write W out
  if (tid < C) {
    const int b = tid >> 4, b0 = b * 16, j = tid & 15;
    float x[16];
#pragma unroll
    for (int rr = 0; rr < 16; ++rr) {
      float acc = (rr == j) ? 1.f : 0.f;
#pragma unroll
      for (int m4 = 0; m4 < rr; m4 += 4) {
        const float4 v4 = lds4(As + (b0 + rr) * kLT + b0 + m4);
        const float v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (m4 + e < rr) acc = fmaf(-v[e], x[m4 + e], acc);
      }
      x[rr] = acc;
    }
#pragma unroll
    for (int rr = 0; rr < 16; ++rr) Ts[(b0 + rr) * kLT + b0 + j] = x[rr];
  } else {
    for (int i = tid - C; i < C * 16; i += kSimtThreads - C) {
      const int r = i >> 4, c = (i & 15) * 4;
      if ((c >> 4) > (r >> 4)) *reinterpret_cast<float4*>(Ts + r * kLT + c) = make_float4(0.f, 0.f, 0.f, 0.f);
      if (a.bwd.TT == nullptr) *reinterpret_cast<float4*>(a.W + mat + i * 4) = lds4(Ws + r * kLT + c);
    }
  }
  __syncthreads();
  // step 2: inside each 32 x 32 diagonal block: T_lo = -D_hi (A_lo D_lo); thread = (block, row, two columns)
  {
    const int s = tid >> 7, r = (tid >> 3) & 15, c0 = (tid & 7) * 2, R0 = 32 * s + 16, C0 = 32 * s;
    float2 p = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float av = As[(R0 + r) * kLT + C0 + k];
      const float2 d = *reinterpret_cast<const float2*>(Ts + (C0 + k) * kLT + C0 + c0);
      p = __ffma2_rn(make_float2(av, av), d, p);
    }
    *reinterpret_cast<float2*>(Ps + (16 * s + r) * LP + c0) = p;
    __syncthreads();
    p = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float tv = -Ts[(R0 + r) * kLT + R0 + k];
      const float2 d = *reinterpret_cast<const float2*>(Ps + (16 * s + k) * LP + c0);
      p = __ffma2_rn(make_float2(tv, tv), d, p);
    }
    *reinterpret_cast<float2*>(Ts + (R0 + r) * kLT + C0 + c0) = p;
  }
  __syncthreads();
  // step 3: T[32:64, 0:32] = -T[32:64, 32:64] (A[32:64, 0:32] T[0:32, 0:32]); thread = (row, four columns)
  {
    const int r = tid >> 3, c0 = (tid & 7) * 4;
    auto row_times = [&](const float* row, float sign, const float* b, int ldb) {
      float2 p0 = make_float2(0.f, 0.f), p1 = p0;
#pragma unroll 8
      for (int k = 0; k < 32; ++k) {
        const float av = sign * row[k];
        const float4 d = lds4(b + k * ldb + c0);
        p0 = __ffma2_rn(make_float2(av, av), make_float2(d.x, d.y), p0);
        p1 = __ffma2_rn(make_float2(av, av), make_float2(d.z, d.w), p1);
      }
      return make_float4(p0.x, p0.y, p1.x, p1.y);
    };
    const float4 p = row_times(As + (32 + r) * kLT, 1.f, Ts, kLT);
    *reinterpret_cast<float4*>(Ps + r * LP + c0) = p;
    __syncthreads();
    const float4 t = row_times(Ts + (32 + r) * kLT + 32, -1.f, Ps, LP);
    *reinterpret_cast<float4*>(Ts + (32 + r) * kLT + c0) = t;
  }
  __syncthreads();
  for (int i = tid; i < C * 16; i += kSimtThreads) {
    const int r = i >> 4, c = (i & 15) * 4;
    *reinterpret_cast<float4*>(a.T + mat + i * 4) = lds4(Ts + r * kLT + c);
    if (a.bwd.TT != nullptr)
      *reinterpret_cast<float4*>(a.bwd.TT + mat + i * 4) = make_float4(Ts[c * kLT + r], Ts[(c + 1) * kLT + r], Ts[(c + 2) * kLT + r], Ts[(c + 3) * kLT + r]);
  }
}

template <int DK> cudaError_t launch_one(const Plan& pl, const IntraArgs& a) {
  const size_t smem = IntraSmem<DK>::bytes(a.in_bf16, a.bwd.TT ? a.dv : 0);
  const cudaError_t e = allow_smem<(int)IntraSmem<DK>::bytes(true, 128)>(intra_simt_kernel<DK>);
  if (e != cudaSuccess) return e;
  return launch_pdl(intra_simt_kernel<DK>, dim3((unsigned)pl.geom.num_slots * pl.p.H), dim3(kSimtThreads), smem, pl.stream, a);
}

}  // namespace

// gates all NULL: the coefficient vectors are in the workspace; else this kernel runs the scan and writes them.
// bwd: the exact backward's extra operands (W is then not written).
cudaError_t launch_intra_simt(const Plan& pl, const void* q, const void* k, const GateArgs& gates, const IntraBwd& bwd, int* launches) {
  IntraArgs a{};
  a.g = pl.geom;
  a.q = q; a.k = k;
  a.in_bf16 = pl.p.io_dtype == MDN_BF16;
  a.coef = reinterpret_cast<float*>(pl.ws + pl.lay.off_coef);
  a.gates = gates;
  a.gp = pl.gp;
  a.scale = pl.p.scale;
  a.T = reinterpret_cast<float*>(pl.ws + pl.lay.off_T);
  a.W = reinterpret_cast<float*>(pl.ws + pl.lay.off_W);
  a.bwd = bwd;
  a.dv = pl.p.dv;
  a.do_bf16 = pl.p.o_dtype == MDN_BF16;
  a.clear_status = pl.clear_status ? reinterpret_cast<int32_t*>(pl.ws + pl.lay.off_status) : nullptr;
  const cudaError_t e = pl.p.dk == 64 ? launch_one<64>(pl, a) : launch_one<128>(pl, a);
  if (e == cudaSuccess) ++*launches;
  return e;
}

}  // namespace mdn
