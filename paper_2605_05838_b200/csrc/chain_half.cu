// a3 + a4 of the plain forward for calls that leave SMs idle: TWO CTAs walk the chunks of one (sequence, head), each with half of
// the value columns.  The same recurrence, products and roundings as chain_tf32.cu (lazily scaled fp32 masters in tensor memory,
// read as tf32; see there); bf16 q/k/v, dk = dv = 128, chunk 64.
//
// What the split buys.  A product costs the same for 64 accumulator lanes as for 128, so half the value columns alone would save
// nothing.  Here the 128 lanes hold BOTH states of the CTA's 64 value columns: of the 32 lanes of a quarter the lower sixteen are
// rows of S^T, the upper sixteen the same rows of M^T.  One product then gives K S and K M (the masters times the K tile), one
// Q S and Q M, and one updates both states: per chunk 16 + 16 products for the state terms and 8 for the updates where chain_tf32.cu
// has 32 (twice as wide) and 16.  What combines S and M terms (R, the output, the rescaling) needs both in one thread: the
// epilogue accesses tensor memory sixteen lanes at a time (16x256b / 16x128b), where a thread gets the same (column, token) of
// both halves, without a shuffle; R^T and V~ stand in both halves of the lanes, so that V~ = T R comes out where either state's
// update operand is made.  The thread layout is that of the warp-level matrix instructions: V comes in and o leaves by
// ldmatrix / stmatrix (transposed).
//
// Per chunk:  MMA-1x X = P K^T (P: both masters)  ->  EPI-1 R^T (bf16 hi + lo) into X  ->  MMA-2 Y = R^T T^T  ->  EPI-2 wS V~ | -wM V~
//             (bf16 hi + lo) into X  ->  MMA-3 P += X K  ->  next chunk's MMA-1x.
// The output runs beside it, on warps of its own, cut to fit the gaps in which the tensor pipe would wait for the epilogue: MMA-1z
// Z = P Q^T partly under EPI-1, partly under EPI-2; o_inter into Z; MMA-3' Z += V~^T W^T behind the NEXT chunk's MMA-1x; output
// tile.  Y and Z are double-buffered for that.
//
// What bounds a chunk: the serial chain of the three product groups (0.72 + 0.36 + 0.51 k cycles), their commit-to-wake latencies
// and the two epilogue steps.  Registers, shared memory and tensor memory (448 of 512 columns) are not the limit; the instruction cache
// is: the warps are in seven roles, all their code is in use at once, and what of it has to be fetched again every chunk is fetched
// through a cache that the SMs of a cluster of SMs share.  So code is kept short: waits are calls (in place: + 23 KB), loops that
// need not be are not unrolled.  A wait in a product-issuing warp costs 0.2 .. 0.4 k cycles even if its phase is long complete: the
// serial chain's products have a warp of their own with three waits per chunk.
//
// Measured: 3.9 .. 4.2 k cycles per chunk against 6.3 k of chain_tf32.cu.  4 x 2048 tokens x 8 heads, whole call: 131.5 -> 94.4 us;
// 200 tokens x 16 heads with a start state: 23.9 -> 18.3.
//
// The layer operations stay with chain_tf32.cu: their output step (a norm over all value columns, so an exchange between the two
// CTAs) kept four output warps busy for longer than a chunk lasts here, and its code made every warp wait for instructions (4 x 3001
// tokens x 16 heads: 252 .. 292 us in four arrangements, 265 there).
#include <cstddef>

#include "chain_tf32.cuh"
#include "mdn_common.cuh"
#include "tc_utils.cuh"

namespace mdn {
namespace {

using namespace tc;

constexpr int kD = 128, kN = 64;   // key columns; value columns of a CTA
// Warps 0..7 epilogue (lane quarter = warp % 4, token half = warp / 4), 8 the products of the state's serial chain, 9 loads of K, V, Q,
// coefficients, 10 the products of the output, 11 loads of T, W, output stores, 12..15 converters, 16..19 output.
constexpr int kEpiWarps = 8, kWarpMma = 8, kWarpLoad = 9, kWarpMmaOut = 10, kWarpStore = 11, kWarpCvt = 12, kCvtWarps = 4, kWarpOut = 16, kOutWarps = 4;
constexpr int kThreads = (kWarpOut + kOutWarps) * 32;
constexpr int kTok = 32, kPk = 16;   // tokens of an epilogue warp; their packed bf16 pairs
constexpr int kZFirst = 4;           // products of MMA-1z that fit under EPI-1, behind MMA-3'

// Shared memory (offsets from a 1024-byte aligned base)
constexpr uint32_t kOffK32 = 0, kOffQ32 = 32768;     // fp32 K and Q [64 tokens x 128 dk]: four dk quarters x [64 rows x 128 B], swizzled
constexpr uint32_t kOffQb = 65536;                   // bf16 Q tile waiting for its copy: two dk halves x [64 rows x 128 B]
constexpr uint32_t kOffOut = 81920, kOutBytes = 16384;   // two output tiles (bf16 or fp32), by the chunk's parity
constexpr uint32_t kOffStage = 114688;               // two stages, by the chunk's parity
constexpr uint32_t kStK = 0, kStV = 16384, kStT = 24576, kStW = 32768, kStCoef = 49152;
constexpr uint32_t kCoefBytes = kChainCoefs * C * sizeof(float);
constexpr uint32_t kStageBytes = 51200;
constexpr uint32_t kTxK = 16384, kTxV = 8192, kTxT = 8192, kTxW = 16384;
constexpr uint32_t kOffAdj = kOffStage + 2 * kStageBytes;
constexpr uint32_t kSmemBytes = kOffAdj + 2 * kAdjBytes + 1024;
static_assert(kStCoef + kCoefBytes <= kStageBytes && kSmemBytes <= kSmemOptin - 4096, "shared-memory layout");

// tensor memory columns: masters P (lanes: S^T | M^T), X, two Y, two Z (by the chunk's parity)
constexpr uint32_t kColP = 0, kColX = 128, kColY = 192, kColZ = 320;
constexpr uint32_t kUpper = 16u << 16;               // the upper sixteen lanes of a warp's quarter: M

// A barrier that a waiter could fall a whole phase behind comes in pairs, by the chunk's parity.  Grouped by their counts: the block's
// first threads set up one each.
struct Bars {
  // one arrival (a commit, or a thread; loads: and their bytes)
  uint64_t kfull[2];  // bf16 K and V tiles of a stage landed
  uint64_t full[2];   // coefficient vectors landed
  uint64_t tfull[2];  // T landed
  uint64_t wfull[2];  // W landed
  uint64_t adj[2];    // a chunk's coefficient block written, its T landed
  uint64_t m3[2];     // masters updated: the stage's K, V, T are free too
  uint64_t mo[2];     // MMA-3' done
  uint64_t ofree[2];  // the output tile has been read by its store
  uint64_t qfull;     // bf16 Q tile landed
  uint64_t mx;        // X done: the fp32 K copy is free too
  uint64_t mz;        // Z done: the fp32 Q copy is free too
  uint64_t m2;        // V~ in Y
  uint64_t fin;       // G after the last chunk written
  // four warps
  uint64_t qfree;     // the bf16 Q tile has been read
  uint64_t q32;       // fp32 Q copy written
  uint64_t oi[2];     // inter-chunk output terms in Z
  uint64_t zu[2];     // Z (the chunk's output) has been read: W is free too
  uint64_t go[2];     // the output tile is staged
  // eight warps
  uint64_t init;      // masters of chunk 0 stored
  uint64_t r;         // EPI-1 done: R^T in X
  uint64_t v;         // MMA-3 may start: update operand in X (eager chunks: masters rescaled)   (+ commit: MMA-1z done)
  uint64_t xr;        // MMA-1x may start: fp32 K copy written (four warps), masters updated (commit)
};
constexpr int kBars1 = 21, kBars4 = kBars1 + 8, kBars8 = kBars4 + 3;
static_assert(offsetof(Bars, qfree) == kBars1 * 8 && offsetof(Bars, init) == kBars4 * 8 && offsetof(Bars, xr) == kBars8 * 8, "barrier groups");

enum Ev : int { kEvTop = 0, kEvXIssued, kEvZIssued, kEvRSeen, kEvM2Issued, kEvMoIssued, kEvVSeen, kEvM3Issued,
                kEvMxSeen, kEvRArrive, kEvOiArrive, kEvM2Seen, kEvVArrive, kEvMoSeen, kEvOutDone, kEvCvtK, kEvCvtKDone, kEvCvtQ,
                kEvCvtQDone, kEvTma, kEvAdj, kEvStored };

template <typename TO>
__global__ void __launch_bounds__(kThreads, 1) chain_half_kernel(const ChainTf32Args a, const __grid_constant__ CUtensorMap map_q,
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

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int H = a.g.H;
  // Coefficients, T and W come from the previous kernel, which lets this one in before it has finished (intra_mma.cu): only
  // the warps that load those wait.  Everything else read here (the call's inputs, the chunk
  // map) was complete before that kernel could let anybody in.  Segment states come from the kernel just before this one.
  const bool early = a.seg_G == 0;
  if (!early) grid_dependency_wait();
  const ChainRun rn = chain_run(a, (int)blockIdx.x >> 1);
  const int v0 = ((int)blockIdx.x & 1) * kN;   // first value column
  const SeqInfo sq = rn.sq;
  const int h = rn.h, nch = sq.nchunks;
  const bool v_zero = rn.v_zero, write_o = rn.write_o;

  const uint32_t s_base = smem_u32(smem);
  auto bar = [](uint64_t& b) { return smem_u32(&b); };

  if (tid == 0) abort_flag = 0;
  if (tid <= kBars8) {
    const bool is_v = tid == kBars8 - 1;
    mbar_init(smem_u32(&bars) + 8 * tid, tid < kBars1 ? 1 : tid < kBars4 ? 4 : tid < kBars8 ? kEpiWarps + (is_v && write_o ? 1 : 0) : kCvtWarps + 1);
    mbar_fence_init();
  }
  static_assert(kCvtWarps == 4 && kOutWarps == 4, "barrier counts");
  if (warp == kWarpMma) tmem_alloc(smem_u32(&tmem_slot), 512);
  if (warp == kWarpLoad && lane == 0) {
    prefetch_tensormap(&map_q); prefetch_tensormap(&map_k); prefetch_tensormap(&map_v);
    prefetch_tensormap(&map_t); prefetch_tensormap(&map_w); prefetch_tensormap(&map_o);
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  bool ok = true;
  volatile int* abortp = &abort_flag;
#define MDN_WAIT(b, par)                                            \
  if (!warp_wait(smem_u32(&bars.b), (par), abortp)) {               \
    ok = false;                                                     \
    break;                                                          \
  }
  // waits on the chain's critical path poll, in place (a call there costs 0.2 k cycles)
#define MDN_POLL(b, par)                                            \
  if (!warp_poll(smem_u32(&bars.b), (par), abortp)) {               \
    ok = false;                                                     \
    break;                                                          \
  }
#ifdef MDN_DEBUG
  // Stamps go to shared memory for the chunks kTlFirst .. kTlFirst + 7 and are copied out when the kernel ends.
  long long* const tline = (blockIdx.x == 0) ? a.timeline : nullptr;
  __shared__ long long tl_sm[kTlChunks][32];
#define MDN_MARK(c, ev) \
  if (tline != nullptr && lane == 0 && (c) >= kTlFirst && (c) < kTlFirst + kTlChunks && \
      ((warp >= kWarpMma && warp <= kWarpCvt) || warp == 2 || warp == kWarpOut)) tl_sm[(c) - kTlFirst][(ev)] = clock64();
  auto now = [&](int i) {   // ... and the nanosecond stamps of the run as a whole in the words before them
    unsigned long long ns;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns));
    if (tline != nullptr && lane == 0) tline[i] = (long long)ns;
  };
#define MDN_NOW(i) now(i)
#else
#define MDN_MARK(c, ev)
#define MDN_NOW(i) (void)0
#endif

  if (warp == 0) { MDN_NOW(0); }
#ifdef MDN_DEBUG
  if (tline != nullptr && tid == 0) {
    uint32_t smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    tline[7] = smid;
  }
#endif
  if (warp == kWarpLoad) {
    // ================================================================== loads, coefficients
    // A stage's K and V tiles are refilled (for chunk c + 2) as soon as MMA-3 has read K, the Q buffer as soon as it is converted.  Who
    // waits for a chunk's coefficient block need not wait for its T.
    int issued = 0;
    float g11 = 1.f, g12 = 0.f, g22 = 1.f;
#pragma unroll 1
    for (int c = 0; c < nch; ++c) {
      const int s = c & 1, tok0 = sq.tok0 + c * C, mat = (sq.slot0 + c) * H + h;
      const uint32_t ph2 = (c >> 1) & 1;
      const uint32_t st = s_base + kOffStage + s * kStageBytes;
      if (c >= 2) MDN_WAIT(m3[s], ph2 ^ 1);
      if (lane == 0) {
        const uint32_t fb = bar(bars.kfull[s]);
        mbar_arrive_expect_tx(fb, kTxK + (v_zero ? 0u : kTxV));
        tma_load_2d(st + kStK, &map_k, h * kD, tok0, fb);
        tma_load_2d(st + kStK + 8192, &map_k, h * kD + 64, tok0, fb);
        if (!v_zero) tma_load_2d(st + kStV, &map_v, h * kD + v0, tok0, fb);
      }
      if (write_o) {
        if (c > 0) MDN_WAIT(qfree, (c - 1) & 1);
        if (lane == 0) {
          mbar_arrive_expect_tx(bar(bars.qfull), kTxK);
          tma_load_2d(s_base + kOffQb, &map_q, h * kD, tok0, bar(bars.qfull));
          tma_load_2d(s_base + kOffQb + 8192, &map_q, h * kD + 64, tok0, bar(bars.qfull));
        }
      }
      if (early && c == 0) { grid_dependency_wait(); MDN_NOW(1); }
      if (lane == 0) {
        const uint32_t fb = bar(bars.full[s]);
        mbar_arrive_expect_tx(fb, kCoefBytes);
        bulk_load(st + kStCoef, a.coef + (size_t)mat * MDN_NUM_COEF * C, kCoefBytes, fb);
      }
      issued = c + 1;
      MDN_MARK(c, kEvTma);
      MDN_WAIT(full[s], ph2);
      MDN_WAIT(tfull[s], ph2);
      if (write_o && c >= 2) MDN_WAIT(oi[s], ph2 ^ 1);   // chunk c - 2's block has been read (MMA-3 of that chunk: by the epilogue)
      publish_coefs<false>(reinterpret_cast<const float*>(smem + kOffStage + s * kStageBytes + kStCoef),
                            reinterpret_cast<float*>(smem + kOffAdj + s * kAdjBytes), a.scale, lane, g11, g12, g22);
      warp_arrive(bar(bars.adj[s]));
      MDN_MARK(c, kEvAdj);
    }
    if (early && nch == 0) grid_dependency_wait();   // (every CTA ends after the previous kernel has)
    if (ok) {
      if (lane == 0) {
        g_final[0] = g11; g_final[1] = g12; g_final[2] = g22;
        mbar_arrive(bar(bars.fin));
      }
    } else if (lane == 0) {   // giving up: let the copies already in flight land before the CTA exits
#pragma unroll 1
      for (int c = max(0, issued - 2); c <= issued; ++c) {   // (of chunk `issued` the first copies may have been issued)
        uint32_t it = 0;
#pragma unroll 1
        while (it < (1u << 18) && !(mbar_try_wait(bar(bars.kfull[c & 1]), (c >> 1) & 1) &&
                                    mbar_try_wait(bar(bars.full[c & 1]), (c >> 1) & 1) &&
                                    (!write_o || mbar_try_wait(bar(bars.qfull), c & 1)))) ++it;
      }
    }
  } else if (warp == kWarpStore) {
    // ================================================================== T and W tiles, output stores
    // (A warp of its own: a copy takes the issuing warp 0.1 .. 0.2 k cycles, and nine a chunk in one warp made the K tile 2 k late.)
    int issued = 0;
    if (early) grid_dependency_wait();
#pragma unroll 1
    for (int c = 0; c < nch + (write_o ? 2 : 0); ++c) {
      const int s = c & 1, mat = (sq.slot0 + c) * H + h;
      const uint32_t ph2 = (c >> 1) & 1;
      const uint32_t st = s_base + kOffStage + s * kStageBytes;
      if (c < nch) {
        if (c >= 2) MDN_WAIT(m3[s], ph2 ^ 1);
        if (lane == 0) {
          mbar_arrive_expect_tx(bar(bars.tfull[s]), kTxT);
          tma_load_2d(st + kStT, &map_t, 0, mat * C, bar(bars.tfull[s]));
        }
        issued = c + 1;
        if (write_o) {
          if (c >= 2) MDN_WAIT(zu[s], ph2 ^ 1);
          if (lane == 0) {
            mbar_arrive_expect_tx(bar(bars.wfull[s]), kTxW);
            tma_load_2d(st + kStW, &map_w, 0, mat * C, bar(bars.wfull[s]));
            tma_load_2d(st + kStW + 8192, &map_w, 32, mat * C, bar(bars.wfull[s]));
          }
        }
      }
      if (c >= 2 && write_o) {
        const int co = c - 2;
        MDN_WAIT(go[s], ph2 ^ 1);
        if (lane == 0) {
          const int n = min(C, sq.len - co * C), tok = sq.tok0 + co * C;
          const uint32_t src = s_base + kOffOut + s * kOutBytes;
          if (n == C) {
            tma_store_2d(&map_o, h * kD + v0, tok, src);
          } else {   // short chunk: rows >= n belong to another sequence; one bulk copy per valid row (an unswizzled tile)
#pragma unroll 1
            for (int r = 0; r < n; ++r)
              bulk_store(static_cast<uint8_t*>(a.o) + (((size_t)(tok + r) * H + h) * kD + v0) * sizeof(TO),
                         src + r * kN * (uint32_t)sizeof(TO), kN * (uint32_t)sizeof(TO));
          }
          tma_store_commit();
          tma_store_wait_read();
          mbar_arrive(bar(bars.ofree[s]));
        }
        MDN_MARK(co, kEvStored);
      }
      __syncwarp();
    }
    if (!ok && lane == 0) {
#pragma unroll 1
      for (int c = max(0, issued - 2); c < issued; ++c) {
        uint32_t it = 0;
#pragma unroll 1
        while (it < (1u << 18) && !(mbar_try_wait(bar(bars.tfull[c & 1]), (c >> 1) & 1) &&
                                    (!write_o || mbar_try_wait(bar(bars.wfull[c & 1]), (c >> 1) & 1)))) ++it;
      }
    }
    if (lane == 0) tma_store_wait_all();
  } else if (warp == kWarpMma) {
    // ================================================================== products of the serial chain
    // The whole warp walks the loop and waits (warp-uniform control flow and operands); one elected lane issues the products and
    // the commits.  A product that reads what another one accumulates waits for that one's commit: MMA-1x issued right behind
    // MMA-3 read masters that lacked part of the update (o off by 3e-4 of its RMS), and was no faster.
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    const uint32_t sb = __shfl_sync(0xffffffffu, s_base, 0);
    const bool lead = elect_one();
    // Column of the bf16 A operands the epilogue leaves in X: K-step k covers tokens 16k .. 16k + 15; the warp that owns those tokens
    // keeps hi (part 0) and lo (part 1) inside its own kTok columns
    auto a_col = [](int part, int k) {
      return static_cast<uint32_t>(kTok * ((16 * k) / kTok) + kPk * part + ((16 * k) % kTok) / 2);
    };
    const uint32_t id64 = idesc_bf16(128, 64, false, false, false);
    const uint32_t id128_mn = idesc_bf16(128, 128, false, true, false);
    const uint32_t id64_tf32 = idesc_tf32(128, 64, false, false, false);
    const uint64_t dK = smem_desc_sw128(sb + kOffK32, 16, 1024);   // + (j >> 2) * 8192 + (j & 3) * 32 bytes per K step
    const uint64_t dT_0 = smem_desc_sw128(sb + kOffStage + kStT, 16, 1024), dT_1 = dT_0 + (kStageBytes >> 4);
    const uint64_t dKmn_0 = smem_desc_sw128(sb + kOffStage + kStK, 8192, 1024), dKmn_1 = dKmn_0 + (kStageBytes >> 4);
#pragma unroll 1
    for (int c = 0; c < nch; ++c) {
      const int s = c & 1;
      const uint32_t ph = c & 1;
      const uint64_t dT = s ? dT_1 : dT_0, dKmn = s ? dKmn_1 : dKmn_0;
      if (c == 0) {
        MDN_WAIT(init, 0);
        if (lane == 0) mbar_arrive(bar(bars.xr));   // (in the place of a previous chunk's commit)
        __syncwarp();
      }
      // ---- MMA-1x: X = P K^T (K S and K M)
      MDN_POLL(xr, ph);
      tc_fence_after_sync();
      if (c == 0) { MDN_NOW(2); }
      MDN_MARK(c, kEvTop);
      if (lead) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          umma_ts_tf32(tm + kColX, tm + kColP + 8 * j, dK + (uint64_t)((j >> 2) * 512 + (j & 3) * 2), id64_tf32, j > 0);
        umma_commit(bar(bars.mx));
      }
      MDN_MARK(c, kEvXIssued);
      // ---- MMA-2: Y = (R_hi + R_lo)^T T^T
      MDN_POLL(r, ph);
      tc_fence_after_sync();
      MDN_MARK(c, kEvRSeen);
      if (lead) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          umma_ts(tm + kColY + 64 * s, tm + kColX + a_col(j >> 2, j & 3), dT + 2 * (j & 3), id64, j > 0);
        umma_commit(bar(bars.m2));
      }
      MDN_MARK(c, kEvM2Issued);
      // ---- MMA-3: P += [wS V~ | -wM V~]^T K   (K tile read MN-major: N = dk, K = tokens)
      MDN_POLL(v, ph);
      tc_fence_after_sync();
      MDN_MARK(c, kEvVSeen);
      if (lead) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
          umma_ts(tm + kColP, tm + kColX + a_col(k >> 2, k & 3), dKmn + 128 * (k & 3), id128_mn, true);
        umma_commit(bar(bars.xr));
        umma_commit(bar(bars.m3[s]));
      }
      MDN_MARK(c, kEvM3Issued);
      if (c == 0) { MDN_NOW(3); }
      if (c == nch - 1) { MDN_NOW(4); }
    }
  } else if (warp == kWarpMmaOut) {
    // ================================================================== products of the output
    // In the gaps of the serial chain: behind MMA-1x the previous chunk's MMA-3' and some of the sixteen products of MMA-1z, behind MMA-2
    // the others (eager chunks: all sixteen first, the masters are rescaled under MMA-2).
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    const uint32_t sb = __shfl_sync(0xffffffffu, s_base, 0);
    const bool lead = elect_one();
    const uint32_t id64_tf32 = idesc_tf32(128, 64, false, false, false);
    const uint64_t dQ = smem_desc_sw128(sb + kOffQ32, 16, 1024);
    const uint64_t dW_0 = smem_desc_sw128(sb + kOffStage + kStW, 16, 1024), dW_1 = dW_0 + (kStageBytes >> 4);
    bool eager = false;
#pragma unroll 1
    for (int c = 0; c <= (write_o ? nch : -1); ++c) {
      const int s = c & 1;
      const uint32_t ph = c & 1, ph2 = (c >> 1) & 1;
      // (waits that are mostly over first, where nothing waits for this warp)
      if (c > 0) {
        MDN_WAIT(wfull[s ^ 1], ((c - 1) >> 1) & 1);
        MDN_WAIT(oi[s ^ 1], ((c - 1) >> 1) & 1);
      }
      if (c < nch) {
        if (c >= 2) MDN_WAIT(zu[s], ph2 ^ 1);   // the output that this chunk's Z held has been read
        MDN_WAIT(adj[s], ph2);
        eager = reinterpret_cast<const float*>(smem + kOffAdj + s * kAdjBytes)[kLazy] == 0.f;
        MDN_WAIT(q32, ph);
        MDN_POLL(mx, ph);
      } else if (eager) {
        MDN_WAIT(m2, ph ^ 1);
      }
      tc_fence_after_sync();
      // ---- MMA-3' of the previous chunk: Z += V~^T W^T, V~ read as tf32 from the accumulator of MMA-2, which another warp issued
      // and whose commit this one has seen: through mx (MMA-1x follows the previous chunk's MMA-3, that its epilogue's wait for
      // m2); behind the last chunk through its own wait for m2, in the middle of MMA-1z or (eager) just above
      if (c > 0) {
        const uint64_t dW = s ? dW_0 : dW_1;
        if (lead) {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            umma_ts_tf32(tm + kColZ + 64 * (s ^ 1), tm + kColY + 64 * (s ^ 1) + 8 * j, dW + (uint64_t)((j >> 2) * 512 + (j & 3) * 2), id64_tf32, true);
          umma_commit(bar(bars.mo[s ^ 1]));
        }
        MDN_MARK(c, kEvMoIssued);
      }
      if (c == nch) break;
      // ---- MMA-1z: Z = P Q^T (Q S and Q M)
      auto mma1z = [&](int j) {
        umma_ts_tf32(tm + kColZ + 64 * s, tm + kColP + 8 * j, dQ + (uint64_t)((j >> 2) * 512 + (j & 3) * 2), id64_tf32, j > 0);
      };
      if (lead) {
#pragma unroll
        for (int j = 0; j < kZFirst; ++j) mma1z(j);
      }
      if (!eager) MDN_POLL(m2, ph);
      if (lead) {
#pragma unroll
        for (int j = kZFirst; j < 16; ++j) mma1z(j);
        umma_commit(bar(bars.mz));
        umma_commit(bar(bars.v));   // MMA-3 may overwrite the masters (and MMA-2 of the next chunk but one what MMA-3' above has read)
      }
      MDN_MARK(c, kEvZIssued);
    }
  } else if (warp >= kWarpCvt && warp < kWarpOut) {
    // ================================================================== converter warps
    // fp32 copies of the K and Q tiles, each as soon as the previous chunk's product has read the one before.
    // A thread takes half a token row (rows across the lanes: minimal wavefronts in both swizzled layouts): the loads first.
    const uint32_t t128 = static_cast<uint32_t>(tid - kWarpCvt * 32), row = t128 & 63, half = t128 >> 6, sw = row & 7;
    auto load8 = [&](uint4 (&u)[8], uint32_t tile) {   // dk half `half`: [64 rows x 128 B]
#pragma unroll
      for (uint32_t i = 0; i < 8; ++i)
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(u[i].x), "=r"(u[i].y), "=r"(u[i].z), "=r"(u[i].w)
                     : "r"(tile + half * 8192 + row * 128 + ((i ^ sw) << 4)));
    };
    // piece i (8 of the half's 64 columns) of the fp32 copy: quarter 2 half + i / 4, 16-byte chunks 2 (i % 4), + 1 of its row
    auto store4 = [&](uint32_t copy, uint32_t i, int e, uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3) {
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                   ::"r"(copy + (2 * half + (i >> 2)) * 8192 + row * 128 + ((((i & 3) * 2 + e) ^ sw) << 4)), "r"(x0), "r"(x1), "r"(x2), "r"(x3)
                   : "memory");
    };
    auto store8 = [&](uint32_t copy, const uint4 (&u)[8]) {
#pragma unroll
      for (uint32_t i = 0; i < 8; ++i) {
        store4(copy, i, 0, u[i].x << 16, u[i].x & 0xffff0000u, u[i].y << 16, u[i].y & 0xffff0000u);
        store4(copy, i, 1, u[i].z << 16, u[i].z & 0xffff0000u, u[i].w << 16, u[i].w & 0xffff0000u);
      }
    };
#pragma unroll 1
    for (int c = 0; c < nch; ++c) {
      const int s = c & 1;
      const uint32_t k_tile = s_base + kOffStage + s * kStageBytes + kStK;
      MDN_WAIT(kfull[s], (c >> 1) & 1);
      if (c > 0) MDN_WAIT(mx, (c - 1) & 1);              // the previous chunk's product has read the copy
      MDN_MARK(c, kEvCvtK);
      uint4 uk[8];
      load8(uk, k_tile);
      store8(s_base + kOffK32, uk);
      fence_proxy_async_smem();
      warp_arrive(bar(bars.xr));
      MDN_MARK(c, kEvCvtKDone);
      if (write_o) {
        MDN_WAIT(qfull, c & 1);
        uint4 uq[8];
        load8(uq, s_base + kOffQb);
        warp_arrive(bar(bars.qfree));
        if (c > 0) MDN_WAIT(mz, (c - 1) & 1);             // the previous chunk's product has read the copy
        MDN_MARK(c, kEvCvtQ);
        store8(s_base + kOffQ32, uq);
        fence_proxy_async_smem();
        warp_arrive(bar(bars.q32));
        MDN_MARK(c, kEvCvtQDone);
      }
    }
  } else if (warp >= kWarpOut) {
    // ================================================================== output warps (one lane quarter each, all 64 tokens)
    const int q4 = warp & 3, row = lane >> 2, cp = 2 * (lane & 3);   // value columns 16 q4 + row, + 8; tokens 32 hf + 8 j + cp, + 1
    const uint32_t tl = tmem + (static_cast<uint32_t>(q4 * 32) << 16);
#pragma unroll 1
    for (int c = 0; c <= (write_o ? nch : -1); ++c) {
      // ---------------- the previous chunk's output: Z -> [64 tokens x 64 value columns] tile in shared memory
      if (c > 0) {
        const int s = (c - 1) & 1, n = min(C, sq.len - (c - 1) * C);
        const uint32_t ph2 = ((c - 1) >> 1) & 1;
        if (c >= 3) MDN_WAIT(ofree[s], ph2 ^ 1);
        MDN_WAIT(mo[s], ph2);
        tc_fence_after_sync();
        MDN_MARK(c - 1, kEvMoSeen);
#pragma unroll 1
        for (int r0 = 0; r0 < C; r0 += 32) {
          uint32_t u[16];
          tmem_ld_16x256_x4(tl + kColZ + 64 * s + r0, u);
          tmem_wait_ld();
          if (sizeof(TO) == 4) {
            float* at = reinterpret_cast<float*>(smem + kOffOut + s * kOutBytes) + (r0 + cp) * kN + 16 * q4 + row;
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
              for (int e = 0; e < 4; ++e) at[(8 * j + (e & 1)) * kN + 8 * (e >> 1)] = __uint_as_float(u[4 * j + e]);
          } else {
            uint32_t pk[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) pk[j] = pack_bf16(__uint_as_float(u[2 * j]), __uint_as_float(u[2 * j + 1]));
            // lane's 16-byte row: token (lane & 7) + 8 (lane >> 4) of a pair of token groups, value columns 8 ((lane >> 3) & 1)
            const uint32_t m_tok = r0 + (lane & 7) + 8 * (lane >> 4), m_ch = 2 * q4 + ((lane >> 3) & 1);
            const uint32_t turn = n == C ? m_tok & 7 : 0;   // (a short chunk leaves row by row)
#pragma unroll
            for (int g = 0; g < 2; ++g)
              stmatrix_x4_trans(s_base + kOffOut + s * kOutBytes + (m_tok + 16 * g) * 128 + ((m_ch ^ turn) << 4), pk + 4 * g);
          }
        }
        tc_fence_before_sync();
        warp_arrive(bar(bars.zu[s]));
        fence_proxy_async_smem();
        warp_arrive(bar(bars.go[s]));
        MDN_MARK(c - 1, kEvOutDone);
      }
      if (c == nch) break;
      // ---------------- inter-chunk output terms cZ .* (Q S) + cU .* (Q M) into the lower lanes of Z, for MMA-3' to accumulate onto
      // (the upper lanes accumulate onto Q M: nobody reads them)
      const int s = c & 1;
      const float* aj = reinterpret_cast<const float*>(smem + kOffAdj + s * kAdjBytes) + cp;
      MDN_WAIT(adj[s], (c >> 1) & 1);
      MDN_WAIT(mz, c & 1);
      tc_fence_after_sync();
#pragma unroll 1
      for (int r0 = 0; r0 < C; r0 += 32) {
        const uint32_t zc = tl + kColZ + 64 * s + r0;
        uint32_t zs[16], zm[16];
        tmem_ld_16x256_x4(zc, zs);
        tmem_ld_16x256_x4(zc + kUpper, zm);
        float2 cz[4], cu[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          cz[j] = *reinterpret_cast<const float2*>(aj + kCz + r0 + 8 * j);
          cu[j] = *reinterpret_cast<const float2*>(aj + kCu + r0 + 8 * j);
        }
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int i = 4 * j + 2 * e;
            const float2 o2 = __ffma2_rn(cz[j], make_float2(__uint_as_float(zs[i]), __uint_as_float(zs[i + 1])),
                                         __fmul2_rn(cu[j], make_float2(__uint_as_float(zm[i]), __uint_as_float(zm[i + 1]))));
            zs[i] = __float_as_uint(o2.x);
            zs[i + 1] = __float_as_uint(o2.y);
          }
        tmem_st_16x256_x4(zc, zs);
      }
      tmem_wait_st();
      tc_fence_before_sync();
      warp_arrive(bar(bars.oi[s]));
      MDN_MARK(c, kEvOiArrive);
    }
  } else if (warp < kEpiWarps) {
    // ================================================================== epilogue warps
    const int q4 = warp & 3, hf = warp >> 2;
    const int r0 = kTok * hf;                      // first token of the per-token steps
    const int row = lane >> 2, cp = 2 * (lane & 3);   // this thread's value columns 16 q4 + row, + 8; tokens r0 + 8 j + cp, + 1
    const uint32_t tl = tmem + (static_cast<uint32_t>(q4 * 32) << 16);
    // ldmatrix / stmatrix: lane's 16-byte row: token (lane & 7) + 8 (lane >> 4) of a pair of token groups, value columns 8 ((lane >> 3) & 1)
    const uint32_t m_tok = r0 + (lane & 7) + 8 * (lane >> 4), m_ch = 2 * q4 + ((lane >> 3) & 1);
    // whole states between global memory and the masters: one lane per row (lower sixteen: S, upper: M)
    const int dg = v0 + 16 * q4 + (lane & 15);
    const bool is_m = lane >= 16;
    // a coefficient vector's values for this thread's four token pairs
    auto coef4 = [&](float2 (&f)[4], const float* aj, int vec) {
#pragma unroll
      for (int j = 0; j < 4; ++j) f[j] = *reinterpret_cast<const float2*>(aj + vec + r0 + 8 * j + cp);
    };
    auto pair = [](const uint32_t (&x)[16], int j, int e) { return make_float2(__uint_as_float(x[4 * j + 2 * e]), __uint_as_float(x[4 * j + 2 * e + 1])); };
    {
      // ---------------- the start state into the masters (all loads in flight at once)
      const float* src = is_m ? rn.M0 : rn.S0;
      const bool id = is_m ? rn.id_m : rn.id_s;
      const int col0 = hf * 64;
      uint32_t x[2][32];
#pragma unroll
      for (int j = 0; j < 64; ++j)
        x[j >> 5][j & 31] = __float_as_uint(src ? __ldg(src + (size_t)(col0 + j) * kD + dg) : (id && col0 + j == dg ? 1.f : 0.f));
      __syncwarp();
      tmem_st32(tl + kColP + col0, x[0]);
      tmem_st32(tl + kColP + col0 + 32, x[1]);
      tmem_wait_st();
      tc_fence_before_sync();
      warp_arrive(bar(bars.init));
    }
#pragma unroll 1
    for (int c = 0; c < nch; ++c) {
      const int s = c & 1;
      const uint32_t ph = c & 1, ph2 = (c >> 1) & 1;
      const float* aj = reinterpret_cast<const float*>(smem + kOffAdj + s * kAdjBytes);
      MDN_WAIT(kfull[s], ph2);
      MDN_WAIT(adj[s], ph2);
      __syncwarp();
      // ---------------- EPI-1: R^T = V^T - cX .* (K S) + cY .* (K M)  -> bf16 hi, lo into X, in both halves of the lanes
      {
        // V and the coefficients are fetched before the wait
        uint32_t vr[8];   // [pair of token groups][m]: token group 2 g + m / 2, value column half m % 2
        if (!v_zero) {
#pragma unroll
          for (int g = 0; g < 2; ++g)
            ldmatrix_x4_trans(s_base + kOffStage + s * kStageBytes + kStV + (m_tok + 16 * g) * 128 + ((m_ch ^ (m_tok & 7)) << 4), vr + 4 * g);
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) vr[i] = 0u;
        }
        float2 cx[4], cy[4];
        coef4(cx, aj, kCx);   // (-cX)
        coef4(cy, aj, kCy);
        MDN_POLL(mx, ph);
        tc_fence_after_sync();
        MDN_MARK(c, kEvMxSeen);
        uint32_t xs[16], xm[16];
        tmem_ld_16x256_x4(tl + kColX + r0, xs);
        tmem_ld_16x256_x4(tl + kUpper + kColX + r0, xm);
        tmem_wait_ld();
        uint32_t hi[8], lo[8];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const uint32_t vw = vr[4 * (j >> 1) + 2 * (j & 1) + e];
            float2 x = make_float2(__uint_as_float(vw << 16), __uint_as_float(vw & 0xffff0000u));
            x = __ffma2_rn(cx[j], pair(xs, j, e), x);
            x = __ffma2_rn(cy[j], pair(xm, j, e), x);
            split_pack_bf16(x, hi[2 * j + e], lo[2 * j + e]);
          }
        // (the columns this warp has just read)
        tmem_st_16x128_x4(tl + kColX + r0, hi);
        tmem_st_16x128_x4(tl + kUpper + kColX + r0, hi);
        tmem_st_16x128_x4(tl + kColX + r0 + kPk, lo);
        tmem_st_16x128_x4(tl + kUpper + kColX + r0 + kPk, lo);
        tmem_wait_st();
      }
      tc_fence_before_sync();
      warp_arrive(bar(bars.r));
      MDN_MARK(c, kEvRArrive);
      // ---------------- eager chunks: the masters take G' = D_c G (under MMA-2) behind MMA-1z, their last reader in this chunk, and the
      // update is added in true coordinates:  Sh <- n11 Sh + n12 Mh, Mh <- n22 Mh
      if (aj[kLazy] == 0.f) {
        if (write_o) MDN_WAIT(mz, ph);
        tc_fence_after_sync();
        const float n11 = aj[kN11], n12 = aj[kN12], n22 = aj[kN22];
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
          const uint32_t col0 = kColP + hf * 64 + i * 32;
          uint32_t ps[16], pm[16];
          tmem_ld_16x256_x4(tl + col0, ps);
          tmem_ld_16x256_x4(tl + kUpper + col0, pm);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            ps[j] = __float_as_uint(unscale_s(n11, __uint_as_float(ps[j]), n12, __uint_as_float(pm[j])));
            pm[j] = __float_as_uint(n22 * __uint_as_float(pm[j]));
          }
          tmem_st_16x256_x4(tl + col0, ps);
          tmem_st_16x256_x4(tl + kUpper + col0, pm);
        }
      }
      // ---------------- EPI-2: wS .* V~ | -wM .* V~ -> X as bf16 hi, lo
      {
        float2 ws[4], wm[4];
        coef4(ws, aj, kWs);
        coef4(wm, aj, kWm);
        MDN_POLL(m2, ph);
        tc_fence_after_sync();
        MDN_MARK(c, kEvM2Seen);
        uint32_t vt[16];
        tmem_ld_16x256_x4(tl + kColY + 64 * s + r0, vt);
        tmem_wait_ld();
        uint32_t hi[8], lo[8];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int e = 0; e < 2; ++e) split_pack_bf16(__fmul2_rn(ws[j], pair(vt, j, e)), hi[2 * j + e], lo[2 * j + e]);
        tmem_st_16x128_x4(tl + kColX + r0, hi);          // X is free: MMA-2 has consumed R
        tmem_st_16x128_x4(tl + kColX + r0 + kPk, lo);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int e = 0; e < 2; ++e)
            split_pack_bf16(__fmul2_rn(make_float2(-wm[j].x, -wm[j].y), pair(vt, j, e)), hi[2 * j + e], lo[2 * j + e]);
        tmem_st_16x128_x4(tl + kUpper + kColX + r0, hi);
        tmem_st_16x128_x4(tl + kUpper + kColX + r0 + kPk, lo);
        tmem_wait_st();
        tc_fence_before_sync();
        warp_arrive(bar(bars.v));
        MDN_MARK(c, kEvVArrive);
      }
    }
    while (ok) {   // (once)
      // ---------------- final states: [S; M] = G [Sh; Mh]
      if (nch > 0) MDN_WAIT(m3[(nch - 1) & 1], ((nch - 1) >> 1) & 1);
      MDN_WAIT(fin, 0);
      __syncwarp();
      const float g11 = g_final[0], g12 = g_final[1], g22 = g_final[2];
      tc_fence_after_sync();
      float* dst = is_m ? rn.Mf : rn.Sf;
#pragma unroll 1
      for (int i = 0; i < 2; ++i) {
        const int col0 = hf * 64 + i * 32;
        uint32_t x[32];
        tmem_ld32(tl + kColP + col0, x);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float mine = __uint_as_float(x[j]), other = __shfl_xor_sync(0xffffffffu, mine, 16);
          const float y = is_m ? g22 * mine : final_s(g11, mine, g12, other);
          if (dst) dst[(size_t)(col0 + j) * kD + dg] = y;
        }
      }
      break;
    }
  }
#undef MDN_WAIT
#undef MDN_POLL
#undef MDN_MARK
  if (warp == 0) { MDN_NOW(6); }

  if (!ok && lane == 0) atomicCAS(a.status, kDevOk, kDevTimeout);
  tc_fence_before_sync();
  __syncthreads();
#ifdef MDN_DEBUG
  if (warp == 0) { MDN_NOW(5); }
  if (tline != nullptr && tid < kTlChunks * 32) tline[(kTlFirst + (tid >> 5)) * 32 + (tid & 31)] = tl_sm[tid >> 5][tid & 31];
#endif
  if (warp == kWarpMma) {
    __syncwarp();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace

cudaError_t launch_chain_half(const Plan& pl, const ChainTf32Args& a, const ChainTensors& in, unsigned items, int* launches) {
  const mdn_params& p = pl.p;
  const uint64_t tokens = (uint64_t)p.B * p.T, mats = (uint64_t)pl.geom.num_slots * p.H, row = (uint64_t)p.H * kD;
  CUtensorMap mq, mk, mv, mt, mw, mo;
  const bool o_bf16 = p.o_dtype == MDN_BF16;
  if (!encode_tma_2d_bf16(&mq, TmaMap2D{in.q, row, tokens, row * 2, 64, 64, true}) ||
      !encode_tma_2d_bf16(&mk, TmaMap2D{in.k, row, tokens, row * 2, 64, 64, true}) ||
      !encode_tma_2d_bf16(&mv, TmaMap2D{in.v, row, tokens, row * 2, kN, 64, true}) ||
      !encode_tma_2d_bf16(&mt, TmaMap2D{pl.ws + pl.lay.off_T, 64, mats * C, 128, 64, 64, true}) ||
      !encode_tma_2d(&mw, TmaMap2D{pl.ws + pl.lay.off_W, 64, mats * C, 256, 32, 64, true}, true) ||
      !encode_tma_2d(&mo, TmaMap2D{a.o, row, tokens, row * (o_bf16 ? 2u : 4u), kN, 64, o_bf16}, !o_bf16))
    return cudaErrorInvalidValue;
  auto kern = o_bf16 ? chain_half_kernel<__nv_bfloat16> : chain_half_kernel<float>;
  cudaError_t e = allow_smem<(int)kSmemBytes>(kern);
  if (e != cudaSuccess) return e;
  e = launch_pdl(kern, dim3(2 * items), dim3(kThreads), kSmemBytes, pl.stream, a, mq, mk, mv, mt, mw, mo);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) ++*launches;
  return e;
}

}  // namespace mdn
