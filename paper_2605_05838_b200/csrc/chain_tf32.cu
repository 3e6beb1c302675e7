// a3 + a4 of the plain forward on the 5th-generation tensor cores (tcgen05, sm_100a), second design: one CTA walks
// the chunks of one (sequence, head) in order; bf16 q/k/v, dk = dv = 128, chunk 64.  (The first design,
// chain_tensor.cu, stays for the training / backward runs.)  Template flag kLayer: the layer's element-wise operations
// of Section 3.3 inside this kernel (q/k norm through the coefficient vectors and the converter warps, RMSNorm and
// sigmoid gate in the output step); kLayer = false compiles them out.
//
// Everything is kept TRANSPOSED: the value dimension (128) is the MMA M dimension and fills the 128 tensor-memory
// lanes, tokens are N (or K).  What is different here:
//
//  * No per-chunk pass over the state.  The fp32 masters S^T, M^T in tensor memory are read by the tensor core as
//    they are, as the A operand of kind::tf32 products (fp32 storage read as tf32), against fp32 copies of the K and
//    Q tiles that two converter warps write one chunk ahead.  No bf16 copy of the state is ever made.
//  * Lazy scaling of the state.  The chunk hand-over  S' = abar_C S - b_C M + dS,  M' = mubar_C M - dM  (state equations
//    below Eq. 12) is a 2 x 2 upper-triangular scalar map D_c on the pair [S; M].  Instead of rescaling the masters
//    every chunk, the masters hold [Sh; Mh] with  [S; M] = G [Sh; Mh],  G = [[g11, g12], [0, g22]]  kept as three
//    scalars:  G' = D_c G  and the update is added in hat coordinates,  [Sh'; Mh'] = [Sh; Mh] + G'^-1 [dS; -dM].
//    Every use of the state then only changes per-token coefficients (all products are linear in the state):
//        K S = g11 (K Sh) + g12 (K Mh),  K M = g22 (K Mh)        ->  R = V - cX .* X + cY .* Y
//        Q S, Q M likewise                                       ->  o_inter = cZ .* Z + cU .* U
//        dS / g11' + (g12' / (g11' g22')) dM,  dM / g22'         ->  per-token weights wS, wM of V~ in the updates
//    with cX = abar g11, cY = (alpha b^-) g22 - abar g12, cZ = scale abar g11, cU = scale (abar g12 - b g22),
//    wS = (gS + (g12'/g22') gM) / g11', wM = gM / g22' (gS = gamma_C eta, gM = (mubar_C/mubar) eta).  The producer
//    warp runs the scalar recurrence of G and writes these six vectors per chunk.  When G' would leave a safe range
//    (g11' or g22' below 2^-64, or |g12'| above g22': fast-decaying gates, mu = 0 tokens, S decaying slower than M) the chunk is "eager":
//    the epilogue warps rescale the masters once by G' (the first design's pre-scaling, with G folded in) and G
//    returns to the identity.  The result is the same recurrence either way; only rounding differs.
//  * One product gives the state terms of the correction AND of the output: B = the K tile stacked on the Q tile
//    (128 rows), so [X | Z] = Sh [K; Q]^T and [Y | U] = Mh [K; Q]^T are two N = 128 products (a product costs the
//    same up to N = 64: measured 45 / 45 / 64 / 128 cycles at N = 32 / 64 / 128 / 256 with A in tensor memory).
//  * The intra-chunk output product reads V~ straight from the accumulator of V~ = T R (kind::tf32 against an fp32 W
//    tile the intra-chunk kernel writes), accumulating onto the inter-chunk terms the epilogue has left there: no
//    operand conversion for it, and it runs under the epilogue's work on the state update.
//
// Per chunk:  MMA-1 [X|Z], [Y|U]  ->  EPI-1 R^T (bf16 hi + lo)  ->  MMA-2 Y = R^T T^T  ->  EPI-2 wS .* V~, wM .* V~ (bf16 hi + lo)
//             ->  MMA-3 Sh^T += (wS V~)^T K, Mh^T -= (wM V~)^T K (K tile read MN-major)  ->  next chunk's MMA-1.
// Off that path: o_inter into U (under MMA-2), MMA-3' U += V~^T W^T (under EPI-2), output tile + TMA store (under MMA-3).
//
// Warps: MMA issuer (one elected lane, tensor-memory owner), TMA producer (also issues the output stores), 8 epilogue
// warps (lane quarter x token half), 2 converter warps.  All hand-offs are mbarriers with bounded waits.
#include <cstdlib>
#include <cstring>

#include "chain_tf32.cuh"
#include "mdn_common.cuh"
#include "tc_utils.cuh"

namespace mdn {
namespace {

using namespace tc;

constexpr int kD = 128;
constexpr int kEpiWarps = 8, kTok = 32, kPk = 16;
// Warp roles: warps 0..7 epilogue (lane quarter = warp % 4, as tensor memory demands), warp 8 MMA issuer, warp 9 TMA producer (it
// also runs the scalar recurrence of G and writes each chunk's coefficient vectors), warps 10, 11 converters
// (fp32 copies of the next chunk's K and Q tiles; they sit on the two schedulers that hold neither the MMA nor the
// TMA warp).  Three warps per scheduler: 168 registers each.  Measured alternatives: the conversion inside the
// epilogue warps (behind the hand-over of the state-update operands) put its 1.5 k cycles of shared-memory traffic
// on the chain's critical path; four converter warps cost the epilogue its registers.
// With the layer operations four more warps (12..15) run the output step's second half, and the register file is split
// by warpgroup: 152 for the epilogue's two, 104 for the other two.  4 x 3001 tokens x 16 heads with q/k norm and output
// step: 298 -> 267 us for the whole call (1 x 2048 x 16: 177 -> 151).
constexpr int kWarpEpi = 0, kWarpMma = 8, kWarpTma = 9, kWarpCvt = 10, kCvtWarps = 2, kWarpOut = 12, kOutWarps = 4;
constexpr int threads_of(bool layer) { return (kEpiWarps + 2 + kCvtWarps + (layer ? kOutWarps : 0)) * 32; }
constexpr int kOutThreads = kOutWarps * 32, kRegEpi = 152, kRegRest = 104;
static_assert(8 * 32 * kRegEpi + 8 * 32 * kRegRest <= 65536, "register file");
constexpr int kEpiThreads = kEpiWarps * 32, kCvtThreads = kCvtWarps * 32;

// shared memory (offsets from a 1024-byte aligned base)
// The K tile is loaded twice: early into a buffer of its own (with the Q tile), where it is free again as soon as
// its fp32 copy is made, so that the next chunk's arrives a whole chunk ahead; and into the stage, where MMA-3 reads
// it (MN-major) at the end of the chunk.  The second load hits the L2.
constexpr uint32_t kOffKQ32 = 0;        // fp32 [K; Q]: four dk quarters x [128 rows (K tokens, then Q tokens) x 128 B], swizzled
constexpr uint32_t kOffCvt = 65536;     // bf16 K and Q tiles waiting for their fp32 copies: [K 16 KB | Q 16 KB], single buffer
constexpr uint32_t kOffStage = 98304;
constexpr uint32_t kStK = 0, kStV = 16384, kStT = 32768, kStW = 40960, kStCoef = 57344;
constexpr uint32_t kCoefBytes = kChainCoefs * C * sizeof(float);
constexpr uint32_t kStageBytes = 59392;
constexpr uint32_t kTxBytes = 2 * 16384 + 8192 + 16384 + kCoefBytes;
constexpr uint32_t kTxW = 16384, kTxV = 16384;   // bytes of the W tile, of the V tile
constexpr uint32_t kStOut = kStV;       // the finished output tile: V area (bf16), V + T + half of W (fp32); all dead by then
constexpr uint32_t kOffAdj = kOffStage + 2 * kStageBytes;
constexpr uint32_t kSmemBytes = kOffAdj + 2 * kAdjBytes + 1024;
static_assert(kStCoef + kCoefBytes <= kStageBytes && kSmemBytes <= 232448, "shared-memory layout");

// tensor memory columns (512 x 128 lanes x 32 bit)
constexpr uint32_t kColS = 0, kColM = 128, kColX = 256, kColZ = 320, kColY = 384, kColU = 448;

struct Bars {
  uint64_t full[2];   // TMA loads of a stage landed                                      (1 + tx bytes)
  uint64_t go[2];     // a stage's output tile is staged and nothing reads the stage any more (256; with the fused output step + 128)
  uint64_t cfull;     // bf16 K, Q of a chunk landed in their buffer                         (1 + tx bytes)
  uint64_t cfree;     // ... and read: the next chunk's may be loaded                       (64)
  uint64_t kq;        // fp32 [K; Q] of a chunk written, the chunk before's Sh update done   (64 + commit)
  uint64_t adj[2];    // a chunk's coefficient block written                              (32)
  uint64_t fin;       // G after the last chunk written                                   (32)
  uint64_t init;      // masters of chunk 0 stored                                        (256)
  uint64_t mx;        // first half of MMA-1 done: X, Z                                    (commit)
  uint64_t m1;        // MMA-1 done: X, Z, Y, U                                            (commit)
  uint64_t r;         // EPI-1 done: R^T hi/lo in X                                        (256)
  uint64_t m2;        // MMA-2 done, inter-chunk output terms stored in U                 (commit + 256; state-only runs: commit)
  uint64_t v1a;       // EPI-2, first part: wS V~ in X (eager chunks: Sh rescaled)         (256)
  uint64_t v1b;       // EPI-2, second part: wM V~ in Y (eager chunks: Mh rescaled)        (256)
  uint64_t m3;        // MMA-3 done, U (the chunk's output) has been read                 (commit + 256; state-only runs: commit)
  uint64_t mo;        // MMA-3' done                                                      (commit)
  uint64_t pn[2];     // fused output step: a stage's fp32 tile is staged                     (256)
};

enum Ev : int { kEvMma1 = 0, kEvM1Seen, kEvRArrive, kEvOiArrive, kEvM2Seen, kEvV1Arrive, kEvOutDone, kEvM3Seen, kEvRSeen,
                kEvV1Seen, kEvCvtStart, kEvCvtDone, kEvTmaIssued, kEvStoresDone, kEvM2Own, kEvEager,
                kEvXzIssued, kEvYuIssued, kEvM2Issued, kEvSIssued, kEvMIssued, kEvV1bSeen, kEvV1bArrive, kEvZuArrive, kEvMoIssued, kEvKqSeen, kEvLoopTop, kEvRArrive2, kEvV1Arrive2 };

template <typename TO> __device__ __forceinline__ void stage_o(uint8_t* tile, int r, int d, float x);
template <> __device__ __forceinline__ void stage_o<float>(uint8_t* tile, int r, int d, float x) {
  reinterpret_cast<float*>(tile)[r * kD + d] = x;
}
template <> __device__ __forceinline__ void stage_o<__nv_bfloat16>(uint8_t* tile, int r, int d, float x) {
  reinterpret_cast<__nv_bfloat16*>(tile)[r * kD + d] = __float2bfloat16_rn(x);
}

template <typename TO, bool kLayer>
__global__ void __launch_bounds__(threads_of(kLayer), 1) chain_tf32_kernel(const ChainTf32Args a, const __grid_constant__ CUtensorMap map_q,
                                                                const __grid_constant__ CUtensorMap map_k,
                                                                const __grid_constant__ CUtensorMap map_v,
                                                                const __grid_constant__ CUtensorMap map_t,
                                                                const __grid_constant__ CUtensorMap map_w,
                                                                const __grid_constant__ CUtensorMap map_o) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) Bars bars;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ float g_final[4];   // G after the last chunk: what the final states are read through
  __shared__ __align__(16) float w_sm[kLayer ? kD : 4];   // RMSNorm weight of the fused output step

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int H = a.g.H;
  // Coefficients, T and W come from the previous kernel, which lets this one in before it has finished (intra_mma.cu): only
  // the producer warp waits, in front of its first load of those.  Everything else read here (the call's inputs, the chunk
  // map) was complete before that kernel could let anybody in.  Segment states come from the kernel just before this one.
  const bool early = a.seg_G == 0;
  if (!early) grid_dependency_wait();
  const ChainRun rn = chain_run(a, (int)blockIdx.x);
  const SeqInfo sq = rn.sq;
  const int h = rn.h, nch = sq.nchunks;
  const float* const S0p = rn.S0;
  const float* const M0p = rn.M0;
  float* const Sfp = rn.Sf;
  float* const Mfp = rn.Mf;
  const bool id_s = rn.id_s, id_m = rn.id_m, v_zero = rn.v_zero, write_o = rn.write_o;

  const uint32_t s_base = smem_u32(smem);
  const uint32_t b_full0 = smem_u32(&bars.full[0]), b_full1 = smem_u32(&bars.full[1]);
  const uint32_t b_go0 = smem_u32(&bars.go[0]), b_go1 = smem_u32(&bars.go[1]);
  const uint32_t b_kq = smem_u32(&bars.kq), b_adj0 = smem_u32(&bars.adj[0]), b_adj1 = smem_u32(&bars.adj[1]);
  const uint32_t b_init = smem_u32(&bars.init), b_m1 = smem_u32(&bars.m1), b_r = smem_u32(&bars.r);
  const uint32_t b_m2 = smem_u32(&bars.m2), b_v1a = smem_u32(&bars.v1a);
  const uint32_t b_v1b = smem_u32(&bars.v1b), b_mx = smem_u32(&bars.mx);
  const uint32_t b_m3 = smem_u32(&bars.m3), b_mo = smem_u32(&bars.mo);
  const uint32_t b_fin = smem_u32(&bars.fin), b_cfull = smem_u32(&bars.cfull), b_cfree = smem_u32(&bars.cfree);
  const uint32_t b_pn0 = smem_u32(&bars.pn[0]), b_pn1 = smem_u32(&bars.pn[1]);
  // kLayer = false compiles the layer operations out
  const bool qk_on = kLayer && a.qk_on;
  const float qk_dh = (qk_on && a.qk_d) ? __ldg(a.qk_d + h) : 0.f;

  if (tid == 0) {
    abort_flag = 0;
    mbar_init(b_full0, 1); mbar_init(b_full1, 1);
    const uint32_t n_go = kEpiThreads + (kLayer && a.post_on && write_o ? kOutThreads : 0);
    mbar_init(b_go0, n_go); mbar_init(b_go1, n_go);
    mbar_init(b_kq, kCvtThreads + 1); mbar_init(b_adj0, 32); mbar_init(b_adj1, 32);
    mbar_init(b_fin, 32); mbar_init(b_cfull, 1); mbar_init(b_cfree, kCvtThreads);
    mbar_init(b_init, kEpiThreads); mbar_init(b_r, kEpiThreads);
    mbar_init(b_v1a, kEpiThreads); mbar_init(b_v1b, kEpiThreads);
    if constexpr (kLayer) { mbar_init(b_pn0, kEpiThreads); mbar_init(b_pn1, kEpiThreads); }
    const uint32_t n_out = 1 + (write_o ? kEpiThreads : 0);
    mbar_init(b_m1, 1); mbar_init(b_m2, n_out); mbar_init(b_m3, n_out); mbar_init(b_mo, 1); mbar_init(b_mx, 1);
    mbar_fence_init();
    mbar_arrive(b_kq);   // (the first chunk has no update before it)
  }
  if (kLayer && tid < kD) w_sm[tid] = (a.post_on && a.post_w) ? __ldg(a.post_w + tid) : 1.f;
  if (warp == kWarpMma) tmem_alloc(smem_u32(&tmem_slot), 512);
  if (warp == kWarpTma && lane == 0) {
    prefetch_tensormap(&map_q); prefetch_tensormap(&map_k); prefetch_tensormap(&map_v);
    prefetch_tensormap(&map_t); prefetch_tensormap(&map_w); prefetch_tensormap(&map_o);
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  bool ok = true;
  volatile int* abortp = &abort_flag;
#define MDN_WAIT(bar, par)                         \
  if (!mbar_wait((bar), (par), abortp)) {          \
    ok = false;                                    \
    break;                                         \
  }
  // waits on the chain's critical path poll without suspending
#define MDN_SPIN(bar, par)                         \
  if (!mbar_wait_spin((bar), (par), abortp)) {     \
    ok = false;                                    \
    break;                                         \
  }
#ifdef MDN_DEBUG
  // Stamps go to shared memory (a global store per stamp slows the stamping thread by hundreds of cycles) for the
  // chunks kTlFirst .. kTlFirst + 7 and are copied out when the kernel ends.
  long long* const tline = (blockIdx.x == 0) ? a.timeline : nullptr;
  __shared__ long long tl_sm[kTlChunks][32];
#define MDN_MARK(c, ev) \
  if (tline != nullptr && lane == 0 && (c) >= kTlFirst && (c) < kTlFirst + kTlChunks && \
      (warp >= kWarpMma || warp == kWarpEpi + 2)) tl_sm[(c) - kTlFirst][(ev)] = clock64();
#define MDN_MARK2(c, ev) \
  if (tline != nullptr && lane == 0 && (c) >= kTlFirst && (c) < kTlFirst + kTlChunks && warp == 5) tl_sm[(c) - kTlFirst][(ev)] = clock64();
#else
#define MDN_MARK(c, ev)
#define MDN_MARK2(c, ev)
#endif

#ifdef MDN_DEBUG
  if (tline != nullptr && tid == 0) {   // clock rate of this run: cycle and nanosecond stamps at both ends
    unsigned long long ns;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns));
    tline[30] = clock64(); tline[31] = (long long)ns;
  }
#endif
  if (warp >= kWarpMma && warp < kWarpOut) {
  if constexpr (kLayer) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegRest));   // (warpgroup 8..11)
  if (warp == kWarpTma) {
    // ================================================================== TMA producer + output stores + coefficients
    // Stage s = c & 1 serves chunk c, then (as the staged output tile) is written out and refilled for chunk c + 2.
    // The whole warp walks the loop; lane 0 issues the copies; every lane writes the coefficients of two tokens.
    {
      int issued = 0, issued_kq = 0;
      float g11 = 1.f, g12 = 0.f, g22 = 1.f;
      for (int c = 0; c < nch + 2; ++c) {
        const int s = c & 1;
        const uint32_t st = s_base + kOffStage + s * kStageBytes;
        if (c < nch) {
          // the chunk's K and Q tiles for the converters first: their buffer is free long before the stage is, and
          // with the fused q/k norm the converters need the head start
          if (c > 0) MDN_WAIT(b_cfree, (c - 1) & 1);   // the previous chunk's bf16 K, Q have been read
          if (lane == 0) {
            const int tok0 = sq.tok0 + c * C;
            mbar_arrive_expect_tx(b_cfull, write_o ? 32768u : 16384u);
            tma_load_2d(s_base + kOffCvt, &map_k, h * kD, tok0, b_cfull);
            tma_load_2d(s_base + kOffCvt + 8192, &map_k, h * kD + 64, tok0, b_cfull);
            if (write_o) {
              tma_load_2d(s_base + kOffCvt + 16384, &map_q, h * kD, tok0, b_cfull);
              tma_load_2d(s_base + kOffCvt + 24576, &map_q, h * kD + 64, tok0, b_cfull);
            }
          }
          __syncwarp();
          issued_kq = c + 1;
        }
        if (c >= 2) {
          const int co = c - 2;
          MDN_WAIT(s ? b_go1 : b_go0, (co >> 1) & 1);
          if (lane == 0) {
            const int n = min(C, sq.len - co * C);
            const int tok0 = sq.tok0 + co * C;
            const uint32_t src = st + kStOut;
            if (!write_o) {
              // Psi / Phi runs of the parallel scan produce states only
            } else if (n == C) {
              tma_store_2d(&map_o, h * kD, tok0, src);
            } else {   // short chunk: rows >= n belong to another sequence; one bulk copy per valid row
              for (int r = 0; r < n; ++r)
                bulk_store(static_cast<uint8_t*>(a.o) + (((size_t)(tok0 + r) * H + h) * kD) * sizeof(TO),
                           src + r * kD * (uint32_t)sizeof(TO), kD * (uint32_t)sizeof(TO));
            }
            tma_store_commit();
            tma_store_wait_read();
          }
          __syncwarp();
          MDN_MARK(co, kEvStoresDone);
        }
        if (c < nch) {
          const uint32_t fb = s ? b_full1 : b_full0;
          if (early && c == 0) grid_dependency_wait();
          if (lane == 0) {
            const int tok0 = sq.tok0 + c * C;
            const int mat = (sq.slot0 + c) * H + h;
            mbar_arrive_expect_tx(fb, kTxBytes - (write_o ? 0u : kTxW) - (v_zero ? kTxV : 0u));
            bulk_load(st + kStCoef, a.coef + (size_t)mat * MDN_NUM_COEF * C, kCoefBytes, fb);
            if (!v_zero) tma_load_2d(st + kStV, &map_v, h * kD, tok0, fb);
            tma_load_2d(st + kStT, &map_t, 0, mat * C, fb);
            if (write_o) {
              tma_load_2d(st + kStW, &map_w, 0, mat * C, fb);
              tma_load_2d(st + kStW + 8192, &map_w, 32, mat * C, fb);
            }
            tma_load_2d(st + kStK, &map_k, h * kD, tok0, fb);          // for MMA-3 at the end of the chunk (L2 hit)
            tma_load_2d(st + kStK + 8192, &map_k, h * kD + 64, tok0, fb);
          }
          __syncwarp();
          MDN_MARK(c, kEvTmaIssued);
          issued = c + 1;
          // ---- the scalar recurrence of G and the chunk's six coefficient vectors (two tokens per lane), as soon as the
          // chunk's coefficient vectors have landed: about a chunk before the epilogue needs them
          MDN_WAIT(fb, (c >> 1) & 1);
          float* aj = reinterpret_cast<float*>(smem + kOffAdj + s * kAdjBytes);
          const float* cf = reinterpret_cast<const float*>(smem + kOffStage + s * kStageBytes + kStCoef);
          publish_coefs<kLayer>(cf, aj, a.scale, lane, g11, g12, g22);
          mbar_arrive(s ? b_adj1 : b_adj0);
        } else if (c == nch) {
          if (early && nch == 0) grid_dependency_wait();   // (every CTA ends after the previous kernel has)
          if (lane == 0) { g_final[0] = g11; g_final[1] = g12; g_final[2] = g22; }
          mbar_arrive(b_fin);
        }
      }
      if (!ok && lane == 0) {   // giving up: let the copies already in flight land before the CTA exits
        for (int c = max(0, issued - 2); c < issued; ++c)
          for (uint32_t it = 0; it < kSpinLimit && !mbar_try_wait((c & 1) ? b_full1 : b_full0, (c >> 1) & 1); ++it) {}
        for (uint32_t it = 0; it < (1u << 16) && issued_kq > 0 && !mbar_try_wait(b_cfull, (issued_kq - 1) & 1); ++it) {}
      }
      if (lane == 0) tma_store_wait_all();
    }
  } else if (warp == kWarpMma) {
    // ================================================================== MMA issuer
    // The whole warp walks the loop and waits (warp-uniform control flow and operands: the descriptors can live in
    // uniform registers); one elected lane issues the products and the commits.
    {
      const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
      const uint32_t sb = __shfl_sync(0xffffffffu, s_base, 0);
      const bool lead = elect_one();
      // Column of the bf16 A operands the epilogue leaves in X, Y: K-step k covers tokens 16k .. 16k + 15; the
      // epilogue warp that owns those tokens keeps hi (part 0) and lo (part 1) inside its own kTok columns
      auto a_col = [](int part, int k) {
        return static_cast<uint32_t>(kTok * ((16 * k) / kTok) + kPk * part + ((16 * k) % kTok) / 2);
      };
      const uint32_t id64 = idesc_bf16(128, 64, false, false, false);
      const uint32_t id128_mn = idesc_bf16(128, 128, false, true, false);
      const uint32_t id128_mn_neg = idesc_bf16(128, 128, false, true, true);
      const uint32_t id1 = idesc_tf32(128, write_o ? 128 : 64, false, false, false);
      const uint32_t id64_tf32 = idesc_tf32(128, 64, false, false, false);
      const uint64_t dKQ = smem_desc_sw128(sb + kOffKQ32, 16, 1024);   // + (j >> 2) * 16384 bytes + (j & 3) * 32 bytes per K step
      // per stage: T, the two halves of W, the K tile read MN-major (+2048 B per 16 tokens)
      const uint64_t dT_0 = smem_desc_sw128(sb + kOffStage + kStT, 16, 1024), dT_1 = dT_0 + (kStageBytes >> 4);
      const uint64_t dW0_0 = smem_desc_sw128(sb + kOffStage + kStW, 16, 1024), dW0_1 = dW0_0 + (kStageBytes >> 4);
      const uint64_t dKmn_0 = smem_desc_sw128(sb + kOffStage + kStK, 8192, 1024), dKmn_1 = dKmn_0 + (kStageBytes >> 4);
      for (int c = 0; c < nch; ++c) {
        const int s = c & 1;
        const uint32_t ph = c & 1;
        const uint64_t dT = s ? dT_1 : dT_0, dW0 = s ? dW0_1 : dW0_0, dW1 = dW0 + (8192 >> 4), dKmn = s ? dKmn_1 : dKmn_0;
        MDN_MARK(c, kEvLoopTop);
        MDN_SPIN(b_kq, ph);
        MDN_MARK(c, kEvKqSeen);
        if (c == 0) MDN_WAIT(b_init, 0);
        // ---- MMA-1: [X | Z] = Sh [K; Q]^T, [Y | U] = Mh [K; Q]^T  (state-only runs: X, Y against K alone).  Each half behind
        // the commit of the update of the master it reads and of the operand it overwrites: products with different
        // accumulators have no order among themselves (one issued right behind another was seen to miss part of what
        // that one accumulates: chain_half.cu).  The tensor pipe stays busy: the Sh update's commit comes while the Mh
        // update runs, that one's while X, Z are made.  Each commit arrives on a barrier that this warp waits for anyway:
        // a wait more costs it 0.15 .. 0.2 k cycles, complete or not, a commit more 0.05 .. 0.1, and it issues for half of
        // the chunk.  (8 x 4096 tokens x 16 heads, 32768 packed x 16: 394.3 -> 394.0, 490.2 -> 491.3 us with this order enforced;
        // with three waits of its own for it 396.7 -> 403.4, 520.7 -> 538.8 on another box.  State-only runs do have a wait more:
        // calls split for the scan take 0 .. 1 % longer, 1 x 30000 x 8 484.5 -> 489.6.)
        tc_fence_after_sync();
        MDN_MARK(c, kEvMma1);
        if (lead) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            umma_ts_tf32(tm + kColX, tm + kColS + 8 * j, dKQ + (uint64_t)((j >> 2) * 1024 + (j & 3) * 2), id1, j > 0);
          umma_commit(b_mx);
        }
        MDN_MARK(c, kEvXzIssued);
        MDN_SPIN(b_m3, ph ^ 1);   // Mh updated, and the previous chunk's output has been read out of U
        tc_fence_after_sync();
        if (lead) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            umma_ts_tf32(tm + kColY, tm + kColM + 8 * j, dKQ + (uint64_t)((j >> 2) * 1024 + (j & 3) * 2), id1, j > 0);
          umma_commit(b_m1);
        }
        MDN_MARK(c, kEvYuIssued);
        // (T, W and the bf16 K tile of the stage have landed: the producer warp waited for them before it published the
        // coefficients the epilogue has used by the time it hands R over)
        // ---- MMA-2: Y = (R_hi + R_lo)^T T^T
        MDN_SPIN(b_r, ph);
        tc_fence_after_sync();
        MDN_MARK(c, kEvRSeen);
        if (lead) {
#pragma unroll
          for (int k = 0; k < 4; ++k) umma_ts(tm + kColY, tm + kColX + a_col(0, k), dT + 2 * k, id64, k > 0);
#pragma unroll
          for (int k = 0; k < 4; ++k) umma_ts(tm + kColY, tm + kColX + a_col(1, k), dT + 2 * k, id64, true);
          umma_commit(b_m2);
        }
        MDN_MARK(c, kEvM2Issued);
        // ---- MMA-3': U += V~^T W^T, V~ read as tf32 from the accumulator of MMA-2 (b_m2: its commit, and U holds the
        // inter-chunk terms), W an fp32 tile.  Runs while the epilogue makes the state-update operands.
        if (write_o) {
          MDN_SPIN(b_m2, ph);
          tc_fence_after_sync();
          MDN_MARK(c, kEvM2Own);
          if (lead) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              umma_ts_tf32(tm + kColU, tm + kColY + 8 * j, ((j >> 2) ? dW1 : dW0) + 2 * (j & 3), id64_tf32, true);
            umma_commit(b_mo);
          }
          MDN_MARK(c, kEvMoIssued);
        }
        // ---- MMA-3: Sh^T += (wS V~)^T K, then Mh^T -= (wM V~)^T K   (K tile read MN-major: N = dk, K = tokens); the
        // first starts while the epilogue still makes the second one's operand
        MDN_SPIN(b_v1a, ph);
        tc_fence_after_sync();
        MDN_MARK(c, kEvV1Seen);
        if (lead) {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            umma_ts(tm + kColS, tm + kColX + a_col(k >> 2, k & 3), dKmn + 128 * (k & 3), id128_mn, true);
          umma_commit(b_kq);
        }
        MDN_MARK(c, kEvSIssued);
        MDN_SPIN(b_v1b, ph);
        tc_fence_after_sync();
        MDN_MARK(c, kEvV1bSeen);
        if (lead) {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            umma_ts(tm + kColM, tm + kColY + a_col(k >> 2, k & 3), dKmn + 128 * (k & 3), id128_mn_neg, true);
          umma_commit(b_m3);
        }
        MDN_MARK(c, kEvMIssued);
      }
    }
  } else {
    // ================================================================== converter warps
    // One chunk ahead of the chain: fp32 copies of the K and Q tiles.  bf16 tile: two dk halves of [64 rows x 128 B];
    // fp32 tile: four dk quarters of [128 rows x 128 B].  A thread takes one token row (rows across the lanes:
    // minimal wavefronts in both swizzled layouts): the sixteen loads of a tile first, then its thirty-two stores.
    const uint32_t row = static_cast<uint32_t>(tid - kWarpCvt * 32), sw = row & 7;
    for (int c = 0; c < nch; ++c) {
      MDN_WAIT(b_cfull, c & 1);
      if (c > 0) MDN_WAIT(b_m1, (c - 1) & 1);   // the previous chunk's products have read the fp32 tiles
      MDN_MARK(c, kEvCvtStart);
      if constexpr (kLayer) {
        // Fused q/k norm: the Q tile's copy is q - d k (fp32, from the two bf16 rows): the output terms then come out of the same
        // products as for a plain q (their 1/|q - d k| rides on the coefficients).  Both rows together, four pieces of each ahead:
        // the next chunk's MMA-1 waits for this (K then Q with K's pieces re-read one by one took 5..6 k cycles).
        const uint32_t src = s_base + kOffCvt + row * 128, dst = s_base + kOffKQ32 + row * 128;
        auto ld = [&](uint4& u, uint32_t at, int c16) {
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                       : "=r"(u.x), "=r"(u.y), "=r"(u.z), "=r"(u.w)
                       : "r"(at + (c16 >> 3) * 8192 + ((static_cast<uint32_t>(c16 & 7) ^ sw) << 4)));
        };
        auto st = [&](uint32_t at, const float (&f)[8], int c16) {
          const uint32_t d0 = at + (c16 >> 2) * 16384, ch = static_cast<uint32_t>((c16 & 3) * 2);
          asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(d0 + ((ch ^ sw) << 4)), "f"(f[0]), "f"(f[1]), "f"(f[2]), "f"(f[3]) : "memory");
          asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(d0 + (((ch + 1) ^ sw) << 4)), "f"(f[4]), "f"(f[5]), "f"(f[6]), "f"(f[7]) : "memory");
        };
        auto widen = [](float (&f)[8], const uint4& u) {
          const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            f[2 * e] = __uint_as_float(w[e] << 16);
            f[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
          }
        };
        uint4 uk[2][4], uq[2][4];
        auto load4 = [&](int p) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            ld(uk[p & 1][i], src, 4 * p + i);
            if (write_o) ld(uq[p & 1][i], src + 16384, 4 * p + i);
          }
        };
        load4(0);
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          if (p < 3) load4(p + 1);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float kf[8], qf[8];
            widen(kf, uk[p & 1][i]);
            st(dst, kf, 4 * p + i);
            if (write_o) {
              widen(qf, uq[p & 1][i]);
#pragma unroll
              for (int e = 0; e < 8; ++e) qf[e] = fmaf(-qk_dh, kf[e], qf[e]);
              st(dst + 64 * 128, qf, 4 * p + i);
            }
          }
        }
      } else {
#pragma unroll 1
        for (int which = 0; which < (write_o ? 2 : 1); ++which) {
          const uint32_t src = s_base + kOffCvt + which * 16384 + row * 128;
          const uint32_t dst = s_base + kOffKQ32 + (which * 64 + row) * 128;
          uint4 u[16];
#pragma unroll
          for (int c16 = 0; c16 < 16; ++c16)
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(u[c16].x), "=r"(u[c16].y), "=r"(u[c16].z), "=r"(u[c16].w)
                         : "r"(src + (c16 >> 3) * 8192 + ((static_cast<uint32_t>(c16 & 7) ^ sw) << 4)));
#pragma unroll
          for (int c16 = 0; c16 < 16; ++c16) {
            const uint32_t d0 = dst + (c16 >> 2) * 16384, ch = static_cast<uint32_t>((c16 & 3) * 2);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(d0 + ((ch ^ sw) << 4)), "r"(u[c16].x << 16),
                         "r"(u[c16].x & 0xffff0000u), "r"(u[c16].y << 16), "r"(u[c16].y & 0xffff0000u) : "memory");
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(d0 + (((ch + 1) ^ sw) << 4)), "r"(u[c16].z << 16),
                         "r"(u[c16].z & 0xffff0000u), "r"(u[c16].w << 16), "r"(u[c16].w & 0xffff0000u) : "memory");
          }
        }
      }
      mbar_arrive(b_cfree);          // the bf16 tiles have been read: the next chunk's may land
      fence_proxy_async_smem();
      mbar_arrive(b_kq);
      MDN_MARK(c, kEvCvtDone);
    }
  }
  } else if (kLayer && warp >= kWarpOut) {
    // ================================================================== output warps
    if constexpr (kLayer) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegRest));   // (warpgroup 12..15)
    // Fused output step, second half: y = sigmoid(g) * o / sqrt(mean_d o^2 + eps) * w_d.  The staged fp32 tile is re-read
    // row-wise, 32 rows at a time: four threads per token sum its 128 squares, rescale and gate.  fp32 output: written back in
    // place (a thread rewrites only the pieces it has read); bf16 output: the final tile goes over the start of the fp32 one,
    // 32 rows over the sixteen before them, once those have been read.  These warps work beside the whole next chunk; when
    // the epilogue warps did this under MMA-1 (2.6 k cycles against its 2.0 k) it delayed every chunk.
    if (a.post_on && write_o) {
      constexpr int kTpr = 4, kPieces = 8;   // threads per token, 16-byte fp32 pieces (8-byte gate pieces) per thread
      // piece i of a row's thread: its columns start at 4 (part + 4 (i ^ row % 4)): the four rows of a half-warp touch different
      // banks, in the fp32 tile (512 bytes a row) and in the bf16 one (256)
      const int t128 = tid - kWarpOut * 32, part = t128 % kTpr;
      int col4[4];   // piece 4 j + r begins at column col4[r] + 64 j
#pragma unroll
      for (int r = 0; r < 4; ++r) col4[r] = 4 * (part + kTpr * (r ^ ((t128 / kTpr) & 3)));
      for (int c = 0; c < nch; ++c) {
        uint8_t* stp = smem + kOffStage + (c & 1) * kStageBytes;
        float* tile = reinterpret_cast<float*>(stp + kStOut);
        uint2 gate[2][kPieces];   // both halves' gates before the wait
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const int prow = 32 * half + t128 / kTpr;
          const __nv_bfloat16* gp = static_cast<const __nv_bfloat16*>(a.post_g) + ((size_t)(sq.tok0 + c * C + prow) * H + h) * kD;
#pragma unroll
          for (int i = 0; i < kPieces; ++i) gate[half][i] = c * C + prow < sq.len ? __ldg(reinterpret_cast<const uint2*>(gp + col4[i & 3] + 64 * (i >> 2))) : make_uint2(0u, 0u);
        }
        uint32_t good = mbar_wait((c & 1) ? b_pn1 : b_pn0, (c >> 1) & 1, abortp) ? 1u : 0u;
        __syncwarp();
        // false (on all four warps: the barrier carries the vote) if that wait ran out
        auto rows32 = [&](int half, const uint2 (&graw)[kPieces]) -> bool {
          const int prow = 32 * half + t128 / kTpr;
          float4 ov[kPieces];
          float ss = 0.f;
#pragma unroll
          for (int i = 0; i < kPieces; ++i) {
            ov[i] = *reinterpret_cast<const float4*>(tile + prow * kD + col4[i & 3] + 64 * (i >> 2));
            ss = fmaf(ov[i].x, ov[i].x, fmaf(ov[i].y, ov[i].y, fmaf(ov[i].z, ov[i].z, fmaf(ov[i].w, ov[i].w, ss))));
          }
          ss += __shfl_xor_sync(0xffffffffu, ss, 1);
          ss += __shfl_xor_sync(0xffffffffu, ss, 2);
          const float rstd = rsqrtf(ss * (1.f / kD) + a.post_eps);
          if (half == 0) {   // these 32 rows have been read (what rows 32..63 turn into lies over rows 16..31)
            asm volatile(
                "{\n\t.reg .pred p, q;\n\t"
                "setp.ne.u32 q, %0, 0;\n\t"
                "barrier.cta.red.and.pred p, 1, %1, q;\n\t"
                "selp.u32 %0, 1, 0, p;\n\t}\n"
                : "+r"(good)
                : "n"(kOutThreads)
                : "memory");
            if (good == 0) return false;
          }
#pragma unroll
          for (int i = 0; i < kPieces; ++i) {
            const int col = col4[i & 3] + 64 * (i >> 2);
            const float4 wv = *reinterpret_cast<const float4*>(w_sm + col);
            const uint2 gr = graw[i];
            const float g0 = __uint_as_float(gr.x << 16), g1 = __uint_as_float(gr.x & 0xffff0000u);
            const float g2 = __uint_as_float(gr.y << 16), g3 = __uint_as_float(gr.y & 0xffff0000u);
            const float y0 = ov[i].x * rstd * wv.x * sigmoid_fast(g0), y1 = ov[i].y * rstd * wv.y * sigmoid_fast(g1);
            const float y2 = ov[i].z * rstd * wv.z * sigmoid_fast(g2), y3 = ov[i].w * rstd * wv.w * sigmoid_fast(g3);
            if (sizeof(TO) == 4) {
              *reinterpret_cast<float4*>(tile + prow * kD + col) = make_float4(y0, y1, y2, y3);
            } else {
              uint2 pk;
              pk.x = pack_bf16(y0, y1); pk.y = pack_bf16(y2, y3);
              *reinterpret_cast<uint2*>(stp + kStOut + (prow * kD + col) * 2) = pk;
            }
          }
          return true;
        };
        ok = rows32(0, gate[0]);
        if (!ok) break;
        rows32(1, gate[1]);
        fence_proxy_async_smem();
        mbar_arrive((c & 1) ? b_go1 : b_go0);
      }
    }
  } else {
    // ================================================================== epilogue warps
    if constexpr (kLayer) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegEpi));    // (warpgroups 0..3, 4..7)
    // lane quarter q4 = warp & 3 (value columns 32 q4 .. +31 = this warp's tensor-memory lanes),
    // token half hf = warp >> 2 (tokens 32 hf .. +31 in the per-token steps, dk columns 64 hf .. +63 of the masters)
    const int q4 = warp & 3, hf = (warp - kWarpEpi) >> 2;
    const int d = q4 * 32 + lane;
    const int r0 = kTok * hf;
    const uint32_t tl = tmem + (static_cast<uint32_t>(q4 * 32) << 16);
    const bool post = kLayer && a.post_on && write_o;
    for (int c = 0; c <= nch; ++c) {
      const float* aj = reinterpret_cast<const float*>(smem + kOffAdj + (c & 1) * kAdjBytes);
      if (c == 0) {
        // ---------------- the start state into the masters
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
          const int col0 = hf * 64 + i * 32;
          uint32_t sr[32], mr[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const float unit = (col0 + j == d) ? 1.f : 0.f;
            sr[j] = __float_as_uint(S0p ? __ldg(S0p + (size_t)(col0 + j) * kD + d) : (id_s ? unit : 0.f));
            mr[j] = __float_as_uint(M0p ? __ldg(M0p + (size_t)(col0 + j) * kD + d) : (id_m ? unit : 0.f));
          }
          tmem_st32(tl + kColS + col0, sr);
          tmem_st32(tl + kColM + col0, mr);
        }
        tmem_wait_st();
        tc_fence_before_sync();
        mbar_arrive(b_init);
      }
      if (c == nch) {
        // ---------------- final states: [S; M] = G [Sh; Mh]  (the last chunk's MMA-3 was waited for below)
        MDN_WAIT(b_fin, 0);
        __syncwarp();
        const float g11 = g_final[0], g12 = g_final[1], g22 = g_final[2];
        tc_fence_after_sync();
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
          const int col0 = hf * 64 + i * 32;
          uint32_t sr[32], mr[32];
          tmem_ld32(tl + kColS + col0, sr);
          tmem_ld32(tl + kColM + col0, mr);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const float sv = __uint_as_float(sr[j]), mv = __uint_as_float(mr[j]);
            if (Sfp) Sfp[(size_t)(col0 + j) * kD + d] = final_s(g11, sv, g12, mv);
            if (Mfp) Mfp[(size_t)(col0 + j) * kD + d] = g22 * mv;
          }
        }
        break;
      }
      const uint32_t ph = c & 1;
      uint8_t* stg = smem + kOffStage + (c & 1) * kStageBytes;
      const __nv_bfloat16* sV = reinterpret_cast<const __nv_bfloat16*>(stg + kStV);
      MDN_WAIT((c & 1) ? b_full1 : b_full0, (c >> 1) & 1);
      MDN_WAIT((c & 1) ? b_adj1 : b_adj0, (c >> 1) & 1);
      // ---------------- EPI-1: R^T = V^T - cX .* X + cY .* Y  -> bf16 hi, lo in X
      {
        // V and the coefficients are fetched BEFORE the waits: shared-memory loads issued after a wait would sit on the
        // chain's critical path, behind whatever the converter warps have queued in the shared-memory pipe
        // (token pairs as float2: the per-token arithmetic runs on the packed two-lane fp32 instructions)
        float2 vv[kTok / 2], cf1[kTok / 2];
#pragma unroll
        for (int j = 0; j < kTok; j += 2)
          vv[j >> 1] = v_zero ? make_float2(0.f, 0.f)
                              : make_float2(__bfloat162float(sV[(r0 + j) * kD + d]), __bfloat162float(sV[(r0 + j + 1) * kD + d]));
#pragma unroll
        for (int j = 0; j < kTok; j += 4) {
          const float4 cx = *reinterpret_cast<const float4*>(aj + kCx + r0 + j);   // -cX
          cf1[j >> 1] = make_float2(cx.x, cx.y); cf1[(j >> 1) + 1] = make_float2(cx.z, cx.w);
        }
        MDN_WAIT(b_mx, ph);          // X is there; Y is still being computed
        __syncwarp();
        tc_fence_after_sync();
        {
          uint32_t x[kTok];
          tmem_ld32(tl + kColX + r0, x);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < kTok; j += 2)
            vv[j >> 1] = __ffma2_rn(cf1[j >> 1], make_float2(__uint_as_float(x[j]), __uint_as_float(x[j + 1])), vv[j >> 1]);
        }
#pragma unroll
        for (int j = 0; j < kTok; j += 4) {
          const float4 cy = *reinterpret_cast<const float4*>(aj + kCy + r0 + j);
          cf1[j >> 1] = make_float2(cy.x, cy.y); cf1[(j >> 1) + 1] = make_float2(cy.z, cy.w);
        }
        MDN_WAIT(b_m1, ph);
        __syncwarp();
        tc_fence_after_sync();
        MDN_MARK(c, kEvM1Seen);
        uint32_t hi[kPk], lo[kPk];
        {
          uint32_t y[kTok];
          tmem_ld32(tl + kColY + r0, y);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < kTok; j += 2)
            split_pack_bf16(__ffma2_rn(cf1[j >> 1], make_float2(__uint_as_float(y[j]), __uint_as_float(y[j + 1])), vv[j >> 1]),
                            hi[j >> 1], lo[j >> 1]);
        }
        // hi and lo both go into the columns this warp has just read (its own kTok columns of X)
        tmem_st16(tl + kColX + r0, hi);
        tmem_st16(tl + kColX + r0 + kPk, lo);
        tmem_wait_st();
      }
      tc_fence_before_sync();
      mbar_arrive(b_r);
      MDN_MARK(c, kEvRArrive);
      MDN_MARK2(c, kEvRArrive2);
      // ---------------- inter-chunk output terms cZ .* Z + cU .* U, left in U for MMA-3' to accumulate onto (under MMA-2)
      if (write_o) {
        uint32_t z[kTok], u[kTok];
        tmem_ld32(tl + kColZ + r0, z);
        tmem_ld32(tl + kColU + r0, u);
        float2 cz[kTok / 2], cu[kTok / 2];   // (their loads run while the tensor-memory loads are in flight)
#pragma unroll
        for (int j = 0; j < kTok; j += 4) {
          const float4 a4 = *reinterpret_cast<const float4*>(aj + kCz + r0 + j);
          const float4 b4 = *reinterpret_cast<const float4*>(aj + kCu + r0 + j);
          cz[j >> 1] = make_float2(a4.x, a4.y); cz[(j >> 1) + 1] = make_float2(a4.z, a4.w);
          cu[j >> 1] = make_float2(b4.x, b4.y); cu[(j >> 1) + 1] = make_float2(b4.z, b4.w);
        }
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < kTok; j += 2) {
          const float2 t2 = __fmul2_rn(cu[j >> 1], make_float2(__uint_as_float(u[j]), __uint_as_float(u[j + 1])));
          const float2 o2 = __ffma2_rn(cz[j >> 1], make_float2(__uint_as_float(z[j]), __uint_as_float(z[j + 1])), t2);
          u[j] = __float_as_uint(o2.x); u[j + 1] = __float_as_uint(o2.y);
        }
        tmem_st32(tl + kColU + r0, u);
        tmem_wait_st();
        tc_fence_before_sync();
        mbar_arrive(b_m2);
        MDN_MARK(c, kEvOiArrive);
      }
      // ---------------- EPI-2: wS .* V~ -> X (handed over first), wM .* V~ -> Y, each as bf16 hi, lo.  V~ itself stays
      // in Y for MMA-3' until that product has read it.  Eager chunks: the masters take G' = D_c G here (MMA-1 of this
      // chunk, their last reader, is done) and the update is added in true coordinates.
      const bool eager = aj[kLazy] == 0.f;
      const float n11 = aj[kN11], n12 = aj[kN12], n22 = aj[kN22];
      // (the first operand's weights are fetched before the wait: shared-memory loads issued after it sit on the
      // chain's critical path behind whatever the converter warps have queued)
      float2 wsv[kTok / 2];
#pragma unroll
      for (int j = 0; j < kTok; j += 4) {
        float4 a4;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(a4.x), "=f"(a4.y), "=f"(a4.z), "=f"(a4.w) : "r"(smem_u32(aj + kWs + r0 + j)));
        wsv[j >> 1] = make_float2(a4.x, a4.y); wsv[(j >> 1) + 1] = make_float2(a4.z, a4.w);
      }
      MDN_WAIT(b_m2, ph);
      __syncwarp();
      tc_fence_after_sync();
      MDN_MARK(c, kEvM2Seen);
      {
        uint32_t vt[kTok];
        tmem_ld32(tl + kColY + r0, vt);
        float2 wmv[kTok / 2];   // (their loads run while the tensor-memory load is in flight)
#pragma unroll
        for (int j = 0; j < kTok; j += 4) {
          const float4 b4 = *reinterpret_cast<const float4*>(aj + kWm + r0 + j);
          wmv[j >> 1] = make_float2(b4.x, b4.y); wmv[(j >> 1) + 1] = make_float2(b4.z, b4.w);
        }
        tmem_wait_ld();
        {
          uint32_t sh[kPk], sl[kPk];
#pragma unroll
          for (int j = 0; j < kTok; j += 2)
            split_pack_bf16(__fmul2_rn(wsv[j >> 1], make_float2(__uint_as_float(vt[j]), __uint_as_float(vt[j + 1]))),
                            sh[j >> 1], sl[j >> 1]);
          tmem_st16(tl + kColX + r0, sh);          // X is free: MMA-2 has consumed R
          tmem_st16(tl + kColX + r0 + kPk, sl);
        }
        if (eager) {   // Sh <- n11 Sh + n12 Mh (Mh still the old one)
          MDN_MARK(c, kEvEager);
#pragma unroll 1
          for (int i = 0; i < 2; ++i) {
            const int col0 = hf * 64 + i * 32;
            uint32_t sr[32], mr[32];
            tmem_ld32(tl + kColS + col0, sr);
            tmem_ld32(tl + kColM + col0, mr);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 32; ++j) sr[j] = __float_as_uint(unscale_s(n11, __uint_as_float(sr[j]), n12, __uint_as_float(mr[j])));
            tmem_st32(tl + kColS + col0, sr);
          }
        }
        tmem_wait_st();
        tc_fence_before_sync();
        mbar_arrive(b_v1a);
        MDN_MARK(c, kEvV1Arrive);
        MDN_MARK2(c, kEvV1Arrive2);
        uint32_t mh[kPk], mlo[kPk];
#pragma unroll
        for (int j = 0; j < kTok; j += 2)
          split_pack_bf16(__fmul2_rn(wmv[j >> 1], make_float2(__uint_as_float(vt[j]), __uint_as_float(vt[j + 1]))),
                          mh[j >> 1], mlo[j >> 1]);
        if (write_o) {   // MMA-3' reads V~ from Y: it must be done before Y is overwritten
          MDN_WAIT(b_mo, ph);
          __syncwarp();
          tc_fence_after_sync();
        }
        tmem_st16(tl + kColY + r0, mh);          // own columns of Y
        tmem_st16(tl + kColY + r0 + kPk, mlo);
      }
      if (eager) {   // Mh <- n22 Mh
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
          const int col0 = hf * 64 + i * 32;
          uint32_t mr[32];
          tmem_ld32(tl + kColM + col0, mr);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 32; ++j) mr[j] = __float_as_uint(n22 * __uint_as_float(mr[j]));
          tmem_st32(tl + kColM + col0, mr);
        }
      }
      tmem_wait_st();
      tc_fence_before_sync();
      mbar_arrive(b_v1b);
      MDN_MARK(c, kEvV1bArrive);
      // ---------------- the chunk's output tile (under MMA-3): U -> [64 x 128] tile in the stage's Q / V area
      if (write_o) {   // (MMA-3' was waited for above)
        uint32_t u[kTok];
        tmem_ld32(tl + kColU + r0, u);
        tmem_wait_ld();
        tc_fence_before_sync();
        mbar_arrive(b_m3);
        MDN_MARK(c, kEvZuArrive);
        bool plain_out = true;
        if constexpr (kLayer) plain_out = !post;
        if (plain_out) {
#pragma unroll
          for (int j = 0; j < kTok; ++j) stage_o<TO>(stg + kStOut, r0 + j, d, __uint_as_float(u[j]));
        } else if constexpr (kLayer) {
          // fused output step, first half: the fp32 tile (value columns across the lanes; V, T and half of the W area,
          // all dead by now).  The output warps do the rest.
          float* tile = reinterpret_cast<float*>(stg + kStOut);
#pragma unroll
          for (int j = 0; j < kTok; ++j) tile[(r0 + j) * kD + d] = __uint_as_float(u[j]);
          mbar_arrive((c & 1) ? b_pn1 : b_pn0);
        }
        fence_proxy_async_smem();
        MDN_MARK(c, kEvOutDone);
      }
      // the stage may be refilled once MMA-3, the last reader of its K tile, is done
      MDN_WAIT(b_m3, ph);
      MDN_MARK(c, kEvM3Seen);
      mbar_arrive((c & 1) ? b_go1 : b_go0);
    }
  }
#undef MDN_WAIT
#undef MDN_SPIN
#undef MDN_MARK
#undef MDN_MARK2

  if (!ok && lane == 0) atomicCAS(a.status, kDevOk, kDevTimeout);
  tc_fence_before_sync();
  __syncthreads();
#ifdef MDN_DEBUG
  if (tline != nullptr && tid == 0) {
    unsigned long long ns;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns));
    tline[62] = clock64(); tline[63] = (long long)ns;
  }
  if (tline != nullptr && tid < kTlChunks * 32) tline[(kTlFirst + (tid >> 5)) * 32 + (tid & 31)] = (tid & 31) < 30 ? tl_sm[tid >> 5][tid & 31] : 0;
#endif
  if (warp == kWarpMma) {
    __syncwarp();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace

cudaError_t launch_chain_tf32(const Plan& pl, const void* q, const void* k, const void* v, const float* S0,
                              const float* M0, void* o, float* Sf, float* Mf, int* launches) {
  const mdn_params& p = pl.p;
  const uint64_t tokens = (uint64_t)p.B * p.T;
  const uint64_t mats = (uint64_t)pl.geom.num_slots * p.H;
  CUtensorMap mq, mk, mv, mt, mw, mo;
  const uint64_t row = (uint64_t)p.H * kD;
  if (!encode_tma_2d_bf16(&mq, TmaMap2D{q, row, tokens, row * 2, 64, 64, true}) ||
      !encode_tma_2d_bf16(&mk, TmaMap2D{k, row, tokens, row * 2, 64, 64, true}) ||
      !encode_tma_2d_bf16(&mv, TmaMap2D{v, row, tokens, row * 2, 128, 64, false}) ||
      !encode_tma_2d_bf16(&mt, TmaMap2D{pl.ws + pl.lay.off_T, 64, mats * C, 128, 64, 64, true}) ||
      !encode_tma_2d(&mw, TmaMap2D{pl.ws + pl.lay.off_W, 64, mats * C, 256, 32, 64, true}, true))
    return cudaErrorInvalidValue;
  const bool o_bf16 = p.o_dtype == MDN_BF16;
  if (!encode_tma_2d(&mo, TmaMap2D{o, row, tokens, row * (o_bf16 ? 2u : 4u), 128, 64, false}, !o_bf16))
    return cudaErrorInvalidValue;
  ChainTf32Args a;
  a.g = pl.geom;
  a.coef = reinterpret_cast<const float*>(pl.ws + pl.lay.off_coef);
  a.S0 = S0; a.M0 = M0; a.o = o; a.Sf = Sf; a.Mf = Mf;
  a.status = reinterpret_cast<int32_t*>(pl.ws + pl.lay.off_status);
  a.scale = p.scale;
  a.seg_G = 0; a.seg_phase = 0; a.seg_first = a.seg_mid = a.seg_least = 0;
  a.seg_E = a.seg_Psi = a.seg_PhiS = a.seg_PhiM = nullptr;
  a.qk_on = pl.qk.on; a.qk_d = pl.qk.d;
  a.post_on = pl.post.on; a.post_w = pl.post.w; a.post_g = pl.post.g; a.post_eps = pl.post.eps;
  const bool layer = a.qk_on || a.post_on;
  a.timeline = nullptr;
#ifdef MDN_DEBUG   // debug builds only (-DMDN_DEBUG): the product library reads nothing from the environment
  const char* tl = getenv("MDN_DEBUG_TIMELINE");   // device address of an int64 buffer, [24][32]
  a.timeline = tl ? reinterpret_cast<long long*>(strtoull(tl, nullptr, 0)) : nullptr;
#endif
  const unsigned chains = (unsigned)pl.geom.num_seqs * p.H;
  auto launch = [&](unsigned grid) -> cudaError_t {
    // two CTAs per run while all of them are resident at once (measured at 32 chains: 131.5 -> 94.4 us; above, a second wave of
    // halves would cost 2 x 4.1 k cycles per chunk against 6.3 k)
    if (!layer && half_runs(grid)) return launch_chain_half(pl, a, ChainTensors{q, k, v}, grid, launches);
    auto kern = layer ? (o_bf16 ? chain_tf32_kernel<__nv_bfloat16, true> : chain_tf32_kernel<float, true>)
                      : (o_bf16 ? chain_tf32_kernel<__nv_bfloat16, false> : chain_tf32_kernel<float, false>);
    cudaError_t e = allow_smem<(int)kSmemBytes>(kern);
    if (e != cudaSuccess) return e;
    e = launch_pdl(kern, dim3(grid), dim3(threads_of(layer)), kSmemBytes, pl.stream, a, mq, mk, mv, mt, mw, mo);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) ++*launches;
    return e;
  };
  const int G = pl.lay.segments;
  if (G <= 1) return launch(chains);

  // ---- parallel inter-chunk scan: Psi / Phi of the middle segments, serial combine, then all segments for real
  constexpr size_t kMat = (size_t)kD * kD;
  float* seg = reinterpret_cast<float*>(pl.seg);
  const SegSplit split = choose_segments(p);
  a.seg_G = G;
  a.seg_first = split.first; a.seg_mid = split.mid; a.seg_least = p.segments ? 1 : kSegLeast;
  a.seg_E = seg;
  a.seg_Psi = a.seg_E + (size_t)chains * (G - 1) * 2 * kMat;
  a.seg_PhiS = a.seg_Psi + (size_t)chains * (G - 2) * 2 * kMat;
  a.seg_PhiM = a.seg_PhiS + (size_t)chains * (G - 2) * 2 * kMat;
  a.seg_phase = 1;
  cudaError_t e = launch(chains * (1 + 3 * (G - 2)));
  if (e != cudaSuccess) return e;
  e = launch_seg_combine(pl, G, a.seg_E, a.seg_Psi, a.seg_PhiS, a.seg_PhiM, launches);
  if (e != cudaSuccess) return e;
  a.seg_phase = 3;
  return launch(chains * (G - 1));
}

}  // namespace mdn
