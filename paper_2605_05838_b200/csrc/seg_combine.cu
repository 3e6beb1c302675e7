// Serial combine step of the parallel inter-chunk scan: for every chain, walk its middle segments in order,
//     [S; M]_g = Phi_g [S; M]_{g-1} + Psi_g          (state at the END of segment g = start of segment g + 1)
// with Phi_g = [Phi_SS Phi_SM; Phi_MS Phi_MM] assembled from the two basis runs of the segment (from (I, 0): the
// column blocks Phi_SS, Phi_MS; from (0, I): Phi_SM, Phi_MM) and Psi_g the run from a zero state.  fp32 FMAs: this is
// (G - 2) products of a 256 x 256 by a 256 x dv matrix per chain.
//
// grid = (chains, dv / COLS); block = 256 threads: 8 x 8 tiles of the 256 x COLS result, every sum over the 256 state rows split
// over 64 / COLS lanes (simt_tile.cuh).  COLS = 16; 8 while that makes at most one CTA per SM (nine chains): half the
// arithmetic of a step in every CTA, the same Phi through twice as many of them.  Phi streams through a three-stage ring of 256 x 32 pieces, the previous state's slice
// stays in shared memory (transposed).  Why this tile: with one row of 16 columns per thread a step spent 17 cycles of the
// shared-memory port per 4 of the FMA pipes (18 us a step, 144 us of a 65536-token call with 16 heads).
#include <type_traits>

#include "simt_tile.cuh"

namespace mdn {
namespace {

constexpr int kD = 128, kPiece = 32, kLd = kPiece + 4, kLp = 2 * kD + 4, kStages = 3, kPieces = 2 * kD / kPiece;
constexpr int kStage = 2 * kD * kLd;
template <int COLS> constexpr size_t kSmem = (size_t)(kStages * kStage + COLS * kLp) * sizeof(float);

template <int COLS> __global__ void __launch_bounds__(kSimtThreads, 1) seg_combine_kernel(int G, float* __restrict__ E,
                                                                     const float* __restrict__ Psi,
                                                                     const float* __restrict__ PhiS,
                                                                     const float* __restrict__ PhiM) {
  extern __shared__ __align__(16) float sm[];
  float* prev = sm + kStages * kStage;   // [column][stacked row of the previous state]
  constexpr size_t kMat = (size_t)kD * kD;
  constexpr int SL = 64 / COLS, kOwn = 8 / SL;   // lanes per sum; rows of a tile that a lane ends up with
  const int chain = blockIdx.x, j0 = blockIdx.y * COLS, tid = threadIdx.x;
  const int s = tid % SL, t = tid / SL;
  // rows rt + kRow i, columns 8 ct + j; four slices: a load phase's two rows are four apart; eight: it is 128 bytes of one row
  constexpr int kRow = SL == 4 ? 32 : 1;
  const int rt = SL == 4 ? ((t & 1) << 2) | ((t >> 1) & 3) | (t & 24) : 8 * t, ct = t >> 5;
  float* e_chain = E + (size_t)chain * (G - 1) * 2 * kMat;
  grid_dependency_wait();
  for (int i = tid; i < 2 * kD * COLS; i += kSimtThreads) {   // state at the end of segment 0 (written by its real run)
    const int c = i % COLS, r = i / COLS;
    prev[c * kLp + r] = e_chain[(size_t)r * kD + j0 + c];      // (S, then M: stacked row r lies at r * 128)
  }
  const int total = (G - 2) * kPieces;
  auto fetch = [&](int p) {   // piece p: segment 1 + p / 8, stacked columns 32 (p % 8) ..
    if (p < total) {
      const int m = (p % kPieces) * kPiece;
      const float* src = (m < kD ? PhiS : PhiM) + ((size_t)chain * (G - 2) + p / kPieces) * 2 * kMat + (m & (kD - 1));
      float* dst = sm + (p % kStages) * kStage;
#pragma unroll
      for (int x = 0; x < 2 * kD * kPiece / 4 / kSimtThreads; ++x) {
        const int f = tid + kSimtThreads * x, r = f >> 3, c4 = (f & 7) * 4;
        cp16(dst + r * kLd + c4, src + (size_t)r * kD + c4, true);
      }
    }
    cp_commit();
  };
  fetch(0);
  fetch(1);
  int p = 0;
  for (int g = 1; g <= G - 2; ++g) {
    const float* psi = Psi + ((size_t)chain * (G - 2) + (g - 1)) * 2 * kMat + j0 + 8 * ct;
    float4 add[kOwn][2];   // the lane's share of Psi: rows rt + kRow (kOwn s + e), eight columns
#pragma unroll
    for (int e = 0; e < kOwn; ++e)
#pragma unroll
      for (int x = 0; x < 2; ++x)
        add[e][x] = __ldg(reinterpret_cast<const float4*>(psi + (size_t)(rt + kRow * (kOwn * s + e)) * kD) + x);
    float2 acc[8][8];
    zero2(acc);
#pragma unroll 1
    for (int q = 0; q < kPieces; ++q, ++p) {
      cp_wait<1>();
      __syncthreads();   // piece p is in (and the previous state complete); piece p - 1 has been read
      fetch(p + 2);
      const float* a = sm + (p % kStages) * kStage + rt * kLd;
      const float* b = prev + 8 * ct * kLp + q * kPiece;
      dot_slices<8, 8>(acc, [&](int i) { return a + kRow * i * kLd; }, [&](int j) { return b + j * kLp; }, s, kPiece / 4, SL);
    }
    float v[64];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) v[8 * i + j] = hsum(acc[i][j]);
    reduce_scatter<64, SL>(v, s);
    __syncthreads();   // everyone is done reading the previous state
    float* out = e_chain + (size_t)g * 2 * kMat + j0 + 8 * ct;
#pragma unroll
    for (int e = 0; e < kOwn; ++e) {
      const int r = rt + kRow * (kOwn * s + e);
      const float add8[8] = {add[e][0].x, add[e][0].y, add[e][0].z, add[e][0].w, add[e][1].x, add[e][1].y, add[e][1].z, add[e][1].w};
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        v[8 * e + j] += add8[j];
        prev[(8 * ct + j) * kLp + r] = v[8 * e + j];
      }
      float4* o4 = reinterpret_cast<float4*>(out + (size_t)r * kD);
      o4[0] = make_float4(v[8 * e], v[8 * e + 1], v[8 * e + 2], v[8 * e + 3]);
      o4[1] = make_float4(v[8 * e + 4], v[8 * e + 5], v[8 * e + 6], v[8 * e + 7]);
    }
  }
  cp_wait<0>();
}

}  // namespace

cudaError_t launch_seg_combine(const Plan& pl, int G, float* E, const float* Psi, const float* PhiS,
                               const float* PhiM, int* launches) {
  const unsigned chains = (unsigned)pl.geom.num_seqs * pl.p.H;
  auto run = [&](auto cols) -> cudaError_t {
    constexpr int kCols = decltype(cols)::value;
    cudaError_t e = allow_smem<(int)kSmem<kCols>>(seg_combine_kernel<kCols>);
    if (e != cudaSuccess) return e;
    return launch_pdl(seg_combine_kernel<kCols>, dim3(chains, kD / kCols), dim3(kSimtThreads), kSmem<kCols>, pl.stream, G, E, Psi, PhiS,
                      PhiM);
  };
  cudaError_t e = chains * (kD / 8) <= kSms ? run(std::integral_constant<int, 8>{}) : run(std::integral_constant<int, 16>{});
  if (e == cudaSuccess) ++*launches;
  return e;
}

}  // namespace mdn
