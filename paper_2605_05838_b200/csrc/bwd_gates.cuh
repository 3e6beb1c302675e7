// Gate gradients of one (chunk, head) from the adjoints of its coefficient vectors and of its two masks: the
// recurrences of Eq. 10 in reverse, column i of gamma / m from the last row up, carrying the adjoints of gamma_{r,i} and
// m_{r,i}.  Shared by the chunk-parallel backward on the tensor cores and the exact fp32 one.
#pragma once
#include "mdn_common.cuh"

namespace mdn {

constexpr int kGateThreads = 256;
constexpr int LG = C + 4;     // floats per row of a 64 x 64 fp32 matrix

// vectors of 64 floats in shared memory: the chain's coefficients, the gates, and the adjoints of both
enum Vec : int { vAbar = 0, vB, vP, vGS, vGM, vMubar, vAlpha, vBeta, vMu, vEta, vBprev,
                 vdAbar, vdB, vdP, vdGS, vdGM, vdMubar, vdAlpha, vdBeta, vdMu, vdEta, vRed };

struct GateOut { float* dbeta; float* dlog_alpha; float* dlog_mu; float* deta; };

// vec: the vectors above; dge(r, i), dgm(r, i): the adjoints of the masks Gamma eta and G^- strictly below the diagonal (asked
// for any r, i: what they return elsewhere is not used), dge_diag(i): Gamma eta's on it; scratch: kGateScratch floats.
// Called by all 256 threads after a barrier; tok0_h: index of the chunk's first token in the [token][H] gate arrays.
//
// With D = d gamma_{r,i}, E = d m_{r,i} of column i, from the last row up (g_S, g_M enter in the last row):
//     D = dg + dGeta_{r,i} eta_i,   dg <- alpha_r (D + dG^-_{r,i} eta_i),      E = dm + beta_r D,   dm <- mu_r E
//     d alpha_r += gamma_{r-1,i} (D + dG^- eta_i),  d beta_r += D m_{r,i},  d mu_r += E m_{r-1,i},
//     d eta_i += dGeta gamma_{r,i} + dG^- alpha_r gamma_{r-1,i}
// A thread takes one column and ONE BLOCK OF SIXTEEN ROWS.  Down a block (gamma, m) is a linear map with three scalars
// [[A, Cm], [0, M]] that no column changes, and (dg, dm) goes back through its transpose plus the block's own terms: so
// every block is walked on its own (in registers), the blocks are joined by at most three such maps, and the rows' sums over columns
// are one shuffle reduction of 48 values.  (The 64-row walks this replaces, with gamma, m, D, E as matrices in shared
// memory, took 24 k of the 66 k cycles of a chunk and head in the tensor-core kernel: almost all of it waiting.)
constexpr int kGateScratch = 2 * C + 4 * 4 + 4 * C * 2;

template <class FE, class FD, class FM>
__device__ __forceinline__ void gate_gradients(float* vec, FE dge_at, FD dge_diag, FM dgm_at, float* scratch, int n, size_t tok0_h, int H,
                                               const GateOut& a) {
  auto V = [&](int which) { return vec + which * C; };
  auto tok = [&](int r) { return tok0_h + (size_t)r * H; };
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float2* ends = reinterpret_cast<float2*>(scratch);               // [64]: a column's (gamma, m) at the end of its own block
  float4* maps = reinterpret_cast<float4*>(scratch + 2 * C);       // [4]: A, Cm, M of a block
  float2* terms = reinterpret_cast<float2*>(scratch + 2 * C + 16); // [4][64]: a block's own terms of (dg, dm)
  constexpr int RB = 16;
  const int i = tid & 63, b = tid >> 6, bi = i >> 4, r0 = RB * b;
  const float eta = V(vEta)[i], gd = dge_diag(i);
  // four rows' values of a vector, one 16-byte load (the same address on every lane)
  auto four = [&](int which, int u, float (&x)[4]) {
    const float4 t = *reinterpret_cast<const float4*>(V(which) + r0 + u);
    x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
  };
  {
    float A = 1.f, Cm = 0.f, M = 1.f, g = 0.f, m = 0.f;
#pragma unroll
    for (int u4 = 0; u4 < RB; u4 += 4) {
      float av[4], bv[4], mv[4];
      four(vAlpha, u4, av); four(vBeta, u4, bv); four(vMu, u4, mv);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        M *= mv[e];
        Cm = fmaf(av[e], Cm, bv[e] * M);
        A *= av[e];
        m = r0 + u4 + e == i ? 1.f : m * mv[e];
        g = fmaf(av[e], g, bv[e] * m);          // (stays 0 until the column begins)
      }
    }
    if (bi == b) ends[i] = make_float2(g, m);
    if (i == 0) maps[b] = make_float4(A, Cm, M, 0.f);
  }
  __syncthreads();
  float gam[RB + 1], mm[RB + 1];   // [0]: the row before the block
  gam[0] = mm[0] = 0.f;
  if (b > bi) {
    const float2 e = ends[i];
    float g = e.x, m = e.y;
    for (int q = bi + 1; q < b; ++q) {
      const float4 f = maps[q];
      g = fmaf(f.x, g, f.y * m);
      m *= f.z;
    }
    gam[0] = g; mm[0] = m;
  }
#pragma unroll
  for (int u4 = 0; u4 < RB; u4 += 4) {
    float av[4], bv[4], mv[4];
    four(vAlpha, u4, av); four(vBeta, u4, bv); four(vMu, u4, mv);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int u = u4 + e;
      mm[u + 1] = r0 + u == i ? 1.f : mm[u] * mv[e];
      gam[u + 1] = fmaf(av[e], gam[u], bv[e] * mm[u + 1]);
    }
  }
  float ge[RB], gm[RB];   // the column's mask adjoints (zero outside the mask; loads without branches)
#pragma unroll
  for (int u = 0; u < RB; ++u) {
    const float x = dge_at(r0 + u, i), y = dgm_at(r0 + u, i);
    ge[u] = r0 + u > i ? x : r0 + u == i ? gd : 0.f;
    gm[u] = r0 + u > i ? y : 0.f;
  }
  {   // the block's own terms of (dg, dm)
    float dg = 0.f, dm = 0.f;
#pragma unroll
    for (int u4 = RB - 4; u4 >= 0; u4 -= 4) {
      float av[4], bv[4], mv[4];
      four(vAlpha, u4, av); four(vBeta, u4, bv); four(vMu, u4, mv);
#pragma unroll
      for (int e = 3; e >= 0; --e) {
        const float D = fmaf(ge[u4 + e], eta, dg), E = fmaf(bv[e], D, dm);
        dg = av[e] * fmaf(gm[u4 + e], eta, D);
        dm = mv[e] * E;
      }
    }
    terms[b * C + i] = make_float2(dg, dm);
  }
  __syncthreads();
  float dg = V(vdGS)[i] * eta, dm = V(vdGM)[i] * eta;   // what g_S, g_M give to the last row
  for (int q = 3; q > b; --q) {
    const float4 f = maps[q];
    const float2 t = terms[q * C + i];
    dm = fmaf(f.z, dm, fmaf(f.y, dg, t.y));
    dg = fmaf(f.x, dg, t.x);
  }
  float v[3 * RB];   // the rows' terms of d alpha, d beta, d mu
  float de = 0.f;
#pragma unroll
  for (int u4 = RB - 4; u4 >= 0; u4 -= 4) {
    float av[4], bv[4], mv[4];
    four(vAlpha, u4, av); four(vBeta, u4, bv); four(vMu, u4, mv);
#pragma unroll
    for (int e = 3; e >= 0; --e) {
      const int u = u4 + e;
      const float D = fmaf(ge[u], eta, dg), E = fmaf(bv[e], D, dm), Dm = fmaf(gm[u], eta, D);
      v[3 * u] = gam[u] * Dm;        // (gamma and m are zero before the column begins)
      v[3 * u + 1] = D * mm[u + 1];
      v[3 * u + 2] = E * mm[u];
      de = fmaf(ge[u], gam[u + 1], fmaf(gm[u] * av[e], gam[u], de));
      dg = av[e] * Dm;
      dm = mv[e] * E;
    }
  }
  if (b == 3) de += V(vdGS)[i] * gam[RB] + V(vdGM)[i] * mm[RB];
  // sums over the warp's 32 columns: halving exchange, 48 -> 3 values per lane pair
  {
    int cur = 3 * RB;
#pragma unroll
    for (int off = 16; off > 1; off >>= 1) {
      const bool up = (lane & off) != 0;
      cur >>= 1;
#pragma unroll
      for (int x = 0; x < 3 * RB / 2; ++x) {
        if (x < cur) {
          const float give = up ? v[x] : v[x + cur], keep = up ? v[x + cur] : v[x];
          v[x] = keep + __shfl_xor_sync(0xffffffffu, give, off);
        }
      }
    }
#pragma unroll
    for (int x = 0; x < 3; ++x) v[x] += __shfl_xor_sync(0xffffffffu, v[x], 1);
  }
  if ((lane & 1) == 0) {
    const int r = r0 + (lane >> 1);
    atomicAdd(V(vdAlpha) + r, v[0]);
    atomicAdd(V(vdBeta) + r, v[1]);
    atomicAdd(V(vdMu) + r, v[2]);
  }
  atomicAdd(V(vdEta) + i, de);
  __syncthreads();
  // The three vector recurrences (p_r = alpha_r b_{r-1};  b_r = alpha_r b_{r-1} + beta_r mubar_r;  the cumulative
  // products) in reverse, on one warp with two rows per lane and everything in registers.  Each reverse chain
  // x_{r-1} = d_{r-1} + c_r x_r is a suffix scan of affine maps: the lane's two rows compose to x_{2l} = B + A x_{2l+2},
  // five shuffle steps compose the lanes.
  if (warp == 0) {
    const int e0 = 2 * lane, e1 = e0 + 1;
    auto rev_scan = [&](float& d0, float& d1, float c1, float c2) {   // c1 = c_{e1}, c2 = c_{e1+1} (0 past the end)
      float A = c1 * c2, B = fmaf(c1, d1, d0);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float A2 = __shfl_down_sync(0xffffffffu, A, o), B2 = __shfl_down_sync(0xffffffffu, B, o);
        if (lane + o < 32) { B = fmaf(A, B2, B); A *= A2; }
      }
      float xn = __shfl_down_sync(0xffffffffu, B, 1);
      if (lane == 31) xn = 0.f;
      d1 = fmaf(c2, xn, d1);
      d0 = B;
    };
    const float2 al = *reinterpret_cast<const float2*>(V(vAlpha) + e0), mu = *reinterpret_cast<const float2*>(V(vMu) + e0);
    const float al2 = lane < 31 ? V(vAlpha)[e0 + 2] : 0.f, mu2 = lane < 31 ? V(vMu)[e0 + 2] : 0.f;
    const float2 be = *reinterpret_cast<const float2*>(V(vBeta) + e0), bp = *reinterpret_cast<const float2*>(V(vBprev) + e0);
    const float2 mb = *reinterpret_cast<const float2*>(V(vMubar) + e0), dP = *reinterpret_cast<const float2*>(V(vdP) + e0);
    const float dP2 = lane < 31 ? V(vdP)[e0 + 2] : 0.f;
    float2 dAl = *reinterpret_cast<const float2*>(V(vdAlpha) + e0), dBe = *reinterpret_cast<const float2*>(V(vdBeta) + e0);
    float2 dMu = *reinterpret_cast<const float2*>(V(vdMu) + e0), dAb = *reinterpret_cast<const float2*>(V(vdAbar) + e0);
    float2 dB = *reinterpret_cast<const float2*>(V(vdB) + e0), dMb = *reinterpret_cast<const float2*>(V(vdMubar) + e0);
    const float ab_prev0 = lane > 0 ? V(vAbar)[e0 - 1] : 1.f, mb_prev0 = lane > 0 ? V(vMubar)[e0 - 1] : 1.f;
    const float ab0 = V(vAbar)[e0];
    // p_r = alpha_r b_{r-1}
    dAl.x = fmaf(dP.x, bp.x, dAl.x); dAl.y = fmaf(dP.y, bp.y, dAl.y);
    dB.x = fmaf(dP.y, al.y, dB.x); dB.y = fmaf(dP2, al2, dB.y);
    rev_scan(dB.x, dB.y, al.y, al2);                      // b_r = alpha_r b_{r-1} + beta_r mubar_r
    dAl.x = fmaf(dB.x, bp.x, dAl.x); dAl.y = fmaf(dB.y, bp.y, dAl.y);
    dBe.x = fmaf(dB.x, mb.x, dBe.x); dBe.y = fmaf(dB.y, mb.y, dBe.y);
    dMb.x = fmaf(dB.x, be.x, dMb.x); dMb.y = fmaf(dB.y, be.y, dMb.y);
    rev_scan(dAb.x, dAb.y, al.y, al2);                    // abar_r = alpha_r abar_{r-1},  mubar_r = mu_r mubar_{r-1}
    rev_scan(dMb.x, dMb.y, mu.y, mu2);
    dAl.x = fmaf(dAb.x, ab_prev0, dAl.x); dAl.y = fmaf(dAb.y, ab0, dAl.y);
    dMu.x = fmaf(dMb.x, mb_prev0, dMu.x); dMu.y = fmaf(dMb.y, mb.x, dMu.y);
    const float de0 = V(vdEta)[e0], de1 = V(vdEta)[e1];
    if (e0 < n) {
      const size_t gi = tok(e0);
      a.dbeta[gi] = dBe.x; a.dlog_alpha[gi] = al.x * dAl.x; a.dlog_mu[gi] = mu.x * dMu.x;
      if (a.deta) a.deta[gi] = de0;
    }
    if (e1 < n) {
      const size_t gi = tok(e1);
      a.dbeta[gi] = dBe.y; a.dlog_alpha[gi] = al.y * dAl.y; a.dlog_mu[gi] = mu.y * dMu.y;
      if (a.deta) a.deta[gi] = de1;
    }
  }
}

}  // namespace mdn
