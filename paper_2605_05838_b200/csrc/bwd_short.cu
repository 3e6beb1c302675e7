// Exact backward of SHORT sequences (fp32, any i/o type, dk, dv in {64, 128}): token by token instead of chunk by chunk.
//
// The chunk form (bwd_exact.cu) costs a whole 64-token chunk in four kernels however few tokens there are; here a token costs
// one forward and one adjoint step of a chain, and nothing else.
//
// One WARP owns four value columns of one (sequence, head): lane l holds rows l, l + 32, .. of those columns of S, M and of their
// adjoints GS, GM in registers, sums over rows are warp shuffles.  A CTA is 16 such warps (64 columns); dv = 128 makes a
// cluster of two CTAs.  Forward first, keeping (S, M) every kBlk tokens; then blocks of kBlk tokens in reverse: recompute
// the block, parking S_{t-1}, M_{t-1} of every token in global scratch, and the adjoint steps, last token first:
//     GS += scale q do^T;  dq = scale S_t do;  dbeta = -<GS, M_t>;  GM -= beta GS;  a = GM v~;  deta = -k.a;
//     dv~ = -eta GM^T k = dv;  dalpha = <GS, S_{t-1}> - dv~.(S_{t-1}^T k);  dmu = <GM, M_{t-1}>;
//     dk = -eta a - alpha S_{t-1} dv~;  GS <- alpha (GS - k dv~^T);  GM <- mu GM.
// dq, dk and the gate gradients sum over value columns: every kSum tokens over the CTA's warps, at the end over the cluster's
// CTAs through distributed shared memory, all in a fixed order.  The grid is persistent (at most a CTA per SM), so that the
// scratch is bounded however many sequences there are.  What bounds it: the latency of a token's reductions (43 % of issue slots, 29 % of
// the FMA pipes); with all SMs at work the parked states do reach HBM (2.0 GB written for 1024 chains of 16 tokens in 0.8 ms).
#include <cooperative_groups.h>

#include "mdn_common.cuh"

namespace mdn {
namespace {

namespace cg = cooperative_groups;

constexpr int kCW = 4, kWarps = 16, kNV = kCW * kWarps, kThreads = kWarps * 32;   // columns per warp, warps, columns per CTA
constexpr int kBlk = 8, kSum = 4, kMax = 56;   // tokens per block of parked states, per sum over the warps, per sequence
static_assert(kMax % kBlk == 0 && kBlk % kSum == 0 && kMax <= C, "blocks tile a sequence, which is one chunk");

template <int DK> struct Scratch {   // per CTA
  static constexpr size_t kSlot = (size_t)kWarps * 2 * DK * kCW, kPrev = kMax / kBlk * kSlot, kFloats = kPrev + kBlk * kSlot;
};
template <int DK> struct Smem {   // float offsets
  static constexpr int k = 0, q = k + kMax * DK, v = q + kMax * DK, d_o = v + kMax * kNV, vt = d_o + kMax * kNV, pred = vt + kMax * kNV,
                       gate = pred + kMax * kNV, sum_g = gate + 4 * kMax, part_g = sum_g + 4 * kMax, part_q = part_g + 4 * kSum * kWarps,
                       part_k = part_q + kSum * kWarps * DK, kFloats = part_k + kSum * kWarps * DK;
};

struct ShortArgs {
  ChunkGeom g;
  const void* q; const void* k; const void* v; const void* d_o;
  bool in_bf16, do_bf16;
  const float* beta; const float* log_alpha; const float* log_mu; const float* eta;
  const float* S0; const float* M0; const float* dSf; const float* dMf;
  float scale;
  int dv, limit;
  bool vec;               // the states and their gradients are 16-byte aligned
  float* scratch;
  float* dq; float* dk; float* dv_out;
  float* dbeta; float* dlog_alpha; float* dlog_mu; float* deta;
  float* dS0; float* dM0;
  int32_t* clear_status;  // or NULL: the status word, when this is the call's first kernel
};

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  return x;
}

__device__ __forceinline__ float load_in(const void* p, size_t i, bool bf16) {
  return bf16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(p)[i]) : static_cast<const float*>(p)[i];
}

template <int DK>
__global__ void __launch_bounds__(kThreads, 1) bwd_short_kernel(const ShortArgs a) {
  constexpr int RW = DK / 32;   // rows per lane
  extern __shared__ __align__(16) float sm[];
  using L = Smem<DK>;
  float* ks = sm + L::k;        // once a token is done: its dk, summed over the CTA's columns
  float* qs = sm + L::q;        // ... its dq
  float* vts = sm + L::vt;
  float* preds = sm + L::pred;  // S_{t-1}^T k_t
  float* gts = sm + L::gate;    // alpha, mu, beta, eta
  float* sum_g = sm + L::sum_g; // [token][d beta, d log_alpha, d log_mu, d eta]

  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int H = a.g.H, DV = a.dv, ncb = DV / kNV, cb = blockIdx.x % ncb;
  const int j0 = cb * kNV + wp * kCW, cl = wp * kCW;   // the warp's first column, within dv and within the CTA
  const int chains = a.g.num_seqs * H;
  grid_dependency_wait();
  grid_launch_dependents();
  if (a.clear_status != nullptr && blockIdx.x == 0 && tid < 4) a.clear_status[tid] = 0;
  float* const ck = a.scratch + (size_t)blockIdx.x * Scratch<DK>::kFloats;
  float* const prev = ck + Scratch<DK>::kPrev;

  for (int chain = blockIdx.x / ncb; chain < chains; chain += gridDim.x / ncb) {
    const int seq = chain / H, h = chain % H;
    const SeqInfo sq = seq_info(a.g, seq);
    if (!short_sequence(sq, a.limit)) continue;   // (the same for both CTAs of a cluster)
    const int n = sq.nchunks > 0 ? sq.len : 0;
    const size_t tok_h = (size_t)sq.tok0 * H + h, st_off = (size_t)chain * DK * DV;

    auto load_pair = [&](const float* p0, const float* p1, float (&x)[RW][kCW], float (&y)[RW][kCW]) {
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        const size_t i = st_off + (size_t)(lane + 32 * r) * DV + j0;
        if (a.vec) {
          const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
          const float4 u = p0 ? *reinterpret_cast<const float4*>(p0 + i) : z, w = p1 ? *reinterpret_cast<const float4*>(p1 + i) : z;
          x[r][0] = u.x; x[r][1] = u.y; x[r][2] = u.z; x[r][3] = u.w;
          y[r][0] = w.x; y[r][1] = w.y; y[r][2] = w.z; y[r][3] = w.w;
        } else {
#pragma unroll
          for (int c = 0; c < kCW; ++c) { x[r][c] = p0 ? p0[i + c] : 0.f; y[r][c] = p1 ? p1[i + c] : 0.f; }
        }
      }
    };
    float S[RW][kCW], M[RW][kCW];
    load_pair(a.S0, a.M0, S, M);
    for (int idx = tid; idx < n * DK; idx += kThreads) {
      const size_t i = (tok_h + (size_t)(idx / DK) * H) * DK + idx % DK;
      ks[idx] = load_in(a.k, i, a.in_bf16);
      qs[idx] = load_in(a.q, i, a.in_bf16);
    }
    for (int idx = tid; idx < n * kNV; idx += kThreads) {
      const size_t i = (tok_h + (size_t)(idx / kNV) * H) * DV + cb * kNV + idx % kNV;
      sm[L::v + idx] = load_in(a.v, i, a.in_bf16);
      sm[L::d_o + idx] = load_in(a.d_o, i, a.do_bf16);
    }
    if (tid < n) {
      const size_t gi = tok_h + (size_t)tid * H;
      gts[tid] = expf(a.log_alpha[gi]);
      gts[kMax + tid] = expf(a.log_mu[gi]);
      gts[2 * kMax + tid] = a.beta[gi];
      gts[3 * kMax + tid] = a.eta ? a.eta[gi] : 1.f;
    }
    __syncthreads();

    // one forward token on the warp's columns; vt = v~, pred = S_{t-1}^T k (for the four columns, on every lane)
    auto forward_token = [&](int t, float (&vt)[kCW], float (&pred)[kCW]) {
      float kr[RW];
#pragma unroll
      for (int r = 0; r < RW; ++r) kr[r] = ks[t * DK + lane + 32 * r];
#pragma unroll
      for (int c = 0; c < kCW; ++c) {
        float w = 0.f;
#pragma unroll
        for (int r = 0; r < RW; ++r) w = fmaf(S[r][c], kr[r], w);
        pred[c] = warp_sum(w);
      }
      const float al = gts[t], mu = gts[kMax + t], be = gts[2 * kMax + t], et = gts[3 * kMax + t];
      const float4 v4 = *reinterpret_cast<const float4*>(sm + L::v + t * kNV + cl);
      vt[0] = v4.x - al * pred[0]; vt[1] = v4.y - al * pred[1]; vt[2] = v4.z - al * pred[2]; vt[3] = v4.w - al * pred[3];
#pragma unroll
      for (int r = 0; r < RW; ++r)
#pragma unroll
        for (int c = 0; c < kCW; ++c) {
          const float m_new = mu * M[r][c] - et * kr[r] * vt[c];
          M[r][c] = m_new;
          S[r][c] = al * S[r][c] - be * m_new;
        }
    };
    auto slot = [&](float* base, int i) { return reinterpret_cast<float4*>(base + ((size_t)i * kWarps + wp) * 2 * DK * kCW); };
    auto store_state = [&](float4* dst) {
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        dst[lane + 32 * r] = make_float4(S[r][0], S[r][1], S[r][2], S[r][3]);
        dst[DK + lane + 32 * r] = make_float4(M[r][0], M[r][1], M[r][2], M[r][3]);
      }
    };
    auto load_state = [&](const float4* src, float (&x)[RW][kCW], float (&y)[RW][kCW]) {
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        const float4 u = src[lane + 32 * r], w = src[DK + lane + 32 * r];
        x[r][0] = u.x; x[r][1] = u.y; x[r][2] = u.z; x[r][3] = u.w;
        y[r][0] = w.x; y[r][1] = w.y; y[r][2] = w.z; y[r][3] = w.w;
      }
    };

    // ---- the state before every block (the last block needs no steps behind it)
    const int blocks = (n + kBlk - 1) / kBlk;
    for (int t = 0; t < (blocks - 1) * kBlk + 1 && t < n; ++t) {
      if (t % kBlk == 0) store_state(slot(ck, t / kBlk));
      float vt[kCW], pred[kCW];
      if (t < (blocks - 1) * kBlk) forward_token(t, vt, pred);
    }
    float GS[RW][kCW], GM[RW][kCW];
    load_pair(a.dSf, a.dMf, GS, GM);

    for (int b = blocks - 1; b >= 0; --b) {
      const int tb = b * kBlk, te = min(n, tb + kBlk);
      load_state(slot(ck, b), S, M);
      for (int t = tb; t < te; ++t) {   // recompute, parking the state BEFORE every token
        store_state(slot(prev, t - tb));
        float vt[kCW], pred[kCW];
        forward_token(t, vt, pred);
        if (lane == 0) {
          *reinterpret_cast<float4*>(vts + t * kNV + cl) = make_float4(vt[0], vt[1], vt[2], vt[3]);
          *reinterpret_cast<float4*>(preds + t * kNV + cl) = make_float4(pred[0], pred[1], pred[2], pred[3]);
        }
      }
      __syncwarp();
      float Sp[RW][kCW], Mp[RW][kCW];   // S_{t-1}, M_{t-1}, fetched one token ahead
      load_state(slot(prev, te - 1 - tb), Sp, Mp);
      for (int ts = tb + (te - 1 - tb) / kSum * kSum, t = te - 1; ts >= tb; ts -= kSum) {
        const int tn = t + 1;   // tokens ts .. tn - 1
        for (; t >= ts; --t) {
          const float al = gts[t], mu = gts[kMax + t], be = gts[2 * kMax + t], et = gts[3 * kMax + t];
          const float4 do4 = *reinterpret_cast<const float4*>(sm + L::d_o + t * kNV + cl);
          const float4 vt4 = *reinterpret_cast<const float4*>(vts + t * kNV + cl), pr4 = *reinterpret_cast<const float4*>(preds + t * kNV + cl);
          const float dov[kCW] = {do4.x, do4.y, do4.z, do4.w}, vtv[kCW] = {vt4.x, vt4.y, vt4.z, vt4.w};
          const float prv[kCW] = {pr4.x, pr4.y, pr4.z, pr4.w};
          float* part_q = sm + L::part_q + ((t - ts) * kWarps + wp) * DK;
          float* part_k = sm + L::part_k + ((t - ts) * kWarps + wp) * DK;
          float kr[RW], ar[RW];
          float nb = 0.f, na = 0.f, nm = 0.f, ke = 0.f;
          float wv[kCW] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int r = 0; r < RW; ++r) {
            kr[r] = ks[t * DK + lane + 32 * r];
            const float qr = a.scale * qs[t * DK + lane + 32 * r];
            float dq_r = 0.f, a_r = 0.f;
#pragma unroll
            for (int c = 0; c < kCW; ++c) {
              const float m_t = mu * Mp[r][c] - et * kr[r] * vtv[c];
              const float s_t = al * Sp[r][c] - be * m_t;
              GS[r][c] = fmaf(qr, dov[c], GS[r][c]);
              dq_r = fmaf(s_t, dov[c], dq_r);
              nb = fmaf(GS[r][c], m_t, nb);
              na = fmaf(GS[r][c], Sp[r][c], na);
              GM[r][c] = fmaf(-be, GS[r][c], GM[r][c]);
              nm = fmaf(GM[r][c], Mp[r][c], nm);
              a_r = fmaf(GM[r][c], vtv[c], a_r);
              wv[c] = fmaf(GM[r][c], kr[r], wv[c]);
            }
            part_q[lane + 32 * r] = a.scale * dq_r;
            ar[r] = a_r;
            ke = fmaf(kr[r], a_r, ke);
          }
          float dvt[kCW];
#pragma unroll
          for (int c = 0; c < kCW; ++c) dvt[c] = -et * warp_sum(wv[c]);
          float dp = 0.f;
#pragma unroll
          for (int c = 0; c < kCW; ++c) dp = fmaf(dvt[c], prv[c], dp);
#pragma unroll
          for (int r = 0; r < RW; ++r) {
            float e_r = 0.f;
#pragma unroll
            for (int c = 0; c < kCW; ++c) {
              e_r = fmaf(Sp[r][c], dvt[c], e_r);
              GS[r][c] = al * (GS[r][c] - kr[r] * dvt[c]);
              GM[r][c] *= mu;
            }
            part_k[lane + 32 * r] = -et * ar[r] - al * e_r;
          }
          if (t > tb) load_state(slot(prev, t - 1 - tb), Sp, Mp);
          nb = warp_sum(nb); na = warp_sum(na); nm = warp_sum(nm); ke = warp_sum(ke);
          if (lane == 0) {
            *reinterpret_cast<float4*>(a.dv_out + (tok_h + (size_t)t * H) * DV + j0) = make_float4(dvt[0], dvt[1], dvt[2], dvt[3]);
            *reinterpret_cast<float4*>(sm + L::part_g + ((t - ts) * kWarps + wp) * 4) = make_float4(-nb, al * (na - dp), mu * nm, -ke);
          }
        }
        __syncthreads();   // these tokens are done: their rows of k and q take the sums over the warps
        for (int idx = tid; idx < (tn - ts) * DK; idx += kThreads) {
          const int i = idx / DK, d = idx % DK;
          float s_q = 0.f, s_k = 0.f;
#pragma unroll
          for (int w = 0; w < kWarps; ++w) {
            s_q += sm[L::part_q + (i * kWarps + w) * DK + d];
            s_k += sm[L::part_k + (i * kWarps + w) * DK + d];
          }
          qs[ts * DK + idx] = s_q;
          ks[ts * DK + idx] = s_k;
        }
        for (int idx = tid; idx < (tn - ts) * 4; idx += kThreads) {
          float s = 0.f;
          for (int w = 0; w < kWarps; ++w) s += sm[L::part_g + ((idx >> 2) * kWarps + w) * 4 + (idx & 3)];
          sum_g[ts * 4 + idx] = s;
        }
        __syncthreads();   // the warps' parts have been read
      }
    }
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const size_t i = st_off + (size_t)(lane + 32 * r) * DV + j0;
      auto put = [&](float* dst, const float (&x)[kCW]) {
        if (dst == nullptr) return;
        if (a.vec) {
          *reinterpret_cast<float4*>(dst + i) = make_float4(x[0], x[1], x[2], x[3]);
        } else {
#pragma unroll
          for (int c = 0; c < kCW; ++c) dst[i + c] = x[c];
        }
      };
      put(a.dS0, GS[r]);
      put(a.dM0, GM[r]);
    }

    // ---- dq, dk, gate gradients: the CTAs' sums, tokens shared out over the CTAs
    const float* peer = sm;
    if (ncb == 2) {
      cg::cluster_group cluster = cg::this_cluster();
      cluster.sync();
      peer = cluster.map_shared_rank(sm, cb ^ 1);
    }
    const float* c0 = cb == 0 ? sm : peer;   // (always the first CTA's sum plus the second's)
    const float* c1 = cb == 0 ? peer : sm;
    for (int idx = tid; idx < n * DK; idx += kThreads) {
      const int t = idx / DK;
      if (ncb == 2 && (t & 1) != cb) continue;
      const size_t i = (tok_h + (size_t)t * H) * DK + idx % DK;
      a.dq[i] = ncb == 2 ? c0[L::q + idx] + c1[L::q + idx] : qs[idx];
      a.dk[i] = ncb == 2 ? c0[L::k + idx] + c1[L::k + idx] : ks[idx];
    }
    if (tid < n && (ncb == 1 || (tid & 1) == cb)) {
      const size_t gi = tok_h + (size_t)tid * H;
      auto sum = [&](int e) { const int at = L::sum_g + tid * 4 + e; return ncb == 2 ? c0[at] + c1[at] : sm[at]; };
      a.dbeta[gi] = sum(0); a.dlog_alpha[gi] = sum(1); a.dlog_mu[gi] = sum(2);
      if (a.deta) a.deta[gi] = sum(3);
    }
    if (ncb == 2) cg::this_cluster().sync();   // both have read the other's sums
    else __syncthreads();
  }
}

template <int DK> cudaError_t launch(const ShortArgs& a, int ctas, cudaStream_t stream) {
  constexpr size_t smem = (size_t)Smem<DK>::kFloats * 4;
  const cudaError_t e = allow_smem<(int)smem>(bwd_short_kernel<DK>);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ctas); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)(a.dv / kNV); attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, bwd_short_kernel<DK>, a);
}

}  // namespace

// Which sequences take this kernel: those of up to `limit` tokens, -1 for none.  A token costs 3.2 us at dk = 128 and 1.9 at 64 in every
// wave of CTAs; the chunk form costs 49 (64 x 64, few chains) to 86 us (128 x 128) up to 32 tokens and grows with the number of
// chains.  The limits are where the two meet (us per call, token form / chunk form):
//     CTAs     dk = 128                                  dk = 64
//     < 64     18 tokens: 65 / 85 (dv 128), 63 / 67      24: 47 / 50 (dv 64), 50 / 72 (dv 128)
//     < 96     24: 85 / 106, 83 / 91                     36: 73 / 73, 74 / 95
//     <= 148   40: 149 / 178, 145 / 160                  56: 114 / 115, 117 / 138
//     more     28: 205 / 214 (256 CTAs)                  40: 325 / 374 (512), 168 / 175 (256)
// Packed input, whose lengths only the device knows: where not all tokens together are within the limit, the call needs both forms,
// one after the other, which pays where the CTAs fill the SMs several times (fewer chains by chunks are less time by chunks)
// and the mean length says that the token form takes many: 100 sequences of 8 tokens x 8 heads 420 / 1177 us, x 1 head
// 82 / 174; but 7 sequences of 5 .. 100 tokens x 8 heads 282 / 180.
BwdShort bwd_short_plan(const mdn_params& p) {
  const int ncb = p.dv / kNV;
  const int64_t seqs = p.num_seqs > 0 ? p.num_seqs : p.B, chains = seqs * p.H, ctas = chains * ncb;
  const bool wide = p.dk == 128;
  const int limit = ctas < 64 ? (wide ? 18 : 24) : ctas < 96 ? (wide ? 24 : 36) : ctas <= kSms ? (wide ? 40 : 56) : wide ? 28 : 40;
  const int64_t mean = p.num_seqs == 0 || ctas <= kSms ? 0 : ctas < 3 * kSms ? limit / 2 : limit;
  if (p.T > limit && p.T > mean * seqs) return BwdShort{-1, 0, 0};
  const int grid = (int)(chains < kSms / ncb ? chains : kSms / ncb) * ncb;
  return BwdShort{limit, grid, (uint64_t)grid * (wide ? Scratch<128>::kFloats : Scratch<64>::kFloats) * 4};
}

cudaError_t launch_bwd_short(const Plan& pl, const BwdIo& io, const BwdShort& plan, void* scratch, int* launches) {
  ShortArgs a{};
  a.g = pl.geom;
  a.q = io.q; a.k = io.k; a.v = io.v; a.d_o = io.d_o;
  a.in_bf16 = pl.p.io_dtype == MDN_BF16; a.do_bf16 = pl.p.o_dtype == MDN_BF16;
  a.beta = io.beta; a.log_alpha = io.log_alpha; a.log_mu = io.log_mu; a.eta = io.eta;
  a.S0 = io.S0; a.M0 = io.M0; a.dSf = io.dSf; a.dMf = io.dMf;
  a.scale = pl.p.scale;
  a.dv = pl.p.dv; a.limit = plan.limit;
  uintptr_t at = 0;
  for (const float* x : {io.S0, io.M0, io.dSf, io.dMf, const_cast<const float*>(io.dS0), const_cast<const float*>(io.dM0)})
    at |= reinterpret_cast<uintptr_t>(x);
  a.vec = (at & 15) == 0;
  a.scratch = static_cast<float*>(scratch);
  a.dq = io.dq; a.dk = io.dk; a.dv_out = io.dv;
  a.dbeta = io.dbeta; a.dlog_alpha = io.dlog_alpha; a.dlog_mu = io.dlog_mu; a.deta = io.deta;
  a.dS0 = io.dS0; a.dM0 = io.dM0;
  a.clear_status = pl.clear_status ? reinterpret_cast<int32_t*>(pl.ws + pl.lay.off_status) : nullptr;
  const cudaError_t e = pl.p.dk == 64 ? launch<64>(a, plan.ctas, pl.stream) : launch<128>(a, plan.ctas, pl.stream);
  if (e == cudaSuccess) ++*launches;
  return e;
}

}  // namespace mdn
