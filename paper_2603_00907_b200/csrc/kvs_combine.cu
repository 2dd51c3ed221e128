// Combine of the attention partials that the key ranges of a query row produce.
//
// One warp (half a one where rows are very many) per (query row, unit): the partial maxima, sums and outputs of the row's key ranges
// are merged into the row's softmax normaliser and attention output
//   o_q = sum_j alpha_qj Vsum_j / c_j,  alpha = softmax_j(scale <q, K_j> + ln c_j)   [Eq. attn_def_vec
// with merged slots].  For the observation window the kernel writes what the statistics pass needs
// (per-query constants, o as two bf16 terms); for the decode check the bf16 output.
#include "kvs_internal.h"

namespace {

constexpr int kThreads = 256;

// kLanes lanes (a warp, or half of one) own a query row, each one 128 / kLanes of its channels.
// kBatch: partial outputs of a row that are requested together.  With few rows the kernel is a chain of L2
// round trips, and shorter with eight; with more rows the registers of a batch cost occupancy, and four are better; with very many
// rows half warps, which request 32 bytes a lane at once.  Us a call in eights, in fours and one by one in half warps:
// 1024 rows of 16 ranges 16.5, 18.4, 20.0; 2048 rows of 8 20.1, 21.6, 24.1, of 2 22.9, 23.3, 23.6; 3072 of 3 26.6, 26.5, 27.5; 4096 of
// 4 21.1, 18.8, 21.2; 6144 of 3 30.6, 29.9, 29.4; 8192 of 2 28.5, 27.0, 25.8; 16384 of 1 47.0, 44.7, 41.3; 65536 171, 160, 148.
// (Two or four partials together in half warps: 65536 rows of one range 25-27 us by events, one by one 25.0.)
// The bounds on the CTAs of an SM leave ptxas the registers of a batch (71 in eights, 59 in fours); without them it takes 48 and
// spills, and 256 rows of 16 ranges take 0.7 us longer.
template <int kBatch, int kLanes>
__global__ void __launch_bounds__(kThreads, kBatch == 1 ? 0 : kBatch == 4 ? 4 : 2)
combine_partials(const CombineArgs a, const RoundTable tab) {
  constexpr int kVec = 32 / kLanes;                        // float4 of a lane
  constexpr int kChannels = 4 * kVec;
  kvs_pdl_launch_dependents();
  kvs_pdl_wait();
  const int seq = blockIdx.z;
  const SeqRound sr = tab.s[seq];
  if (sr.n <= 0) return;
  const int unit = sr.b * a.Hkv + blockIdx.y;
  const int m_own = blockIdx.x * (kThreads / kLanes) + (int)threadIdx.x / kLanes;
  const int lane = threadIdx.x % kLanes;
  if (m_own >= a.M && lane == 0 && a.qc2 && m_own < a.M_pad) {
    // padding rows of the per-query constants: alpha = exp2(-inf) = 0
    float* qc = a.qc2 + ((size_t)unit * a.M_pad + m_own) * 2 - (m_own & 1);
    qc[0] = -INFINITY;
    qc[2] = 0.f;
  }
  if (m_own / (32 / kLanes) * (32 / kLanes) >= a.M) return;   // (the whole warp)
  const bool mine = m_own < a.M;                           // (else the lanes keep the row beside company)
  const int m = mine ? m_own : a.M - 1;
  const size_t base = (size_t)unit * a.splits * a.M + m;
  const float2* ml = a.part_ml + base;
  const float4* po_row = reinterpret_cast<const float4*>(a.part_o + base * KVS_D) + kVec * lane;
  const size_t po_step = (size_t)a.M * (KVS_D / 4);
  const float2 first = lane < a.splits ? ml[(size_t)lane * a.M] : make_float2(-INFINITY, 0.f);
  float mstar = first.x, Z = 0.f;
  float acc[kChannels] = {};
  for (int s = kLanes + lane; s < a.splits; s += kLanes) mstar = fmaxf(mstar, ml[(size_t)s * a.M].x);
#pragma unroll
  for (int k = kLanes / 2; k > 0; k >>= 1) mstar = fmaxf(mstar, __shfl_xor_sync(0xffffffffu, mstar, k));
  for (int s0 = 0; s0 < a.splits; s0 += kLanes) {
    const int cnt = min(kLanes, a.splits - s0);
    float2 own = first;
    if (s0 > 0) own = lane < cnt ? ml[(size_t)(s0 + lane) * a.M] : make_float2(-INFINITY, 0.f);
    const float f = own.x == -INFINITY ? 0.f : fast_exp2(own.x - mstar);
    // An empty range has left no output: what stands there is read and dropped (a condition on a load is waited for
    // before it).  One of weight 0 counts: 0 times infinity stays NaN.
    const uint32_t filled = __ballot_sync(0xffffffffu, own.x != -INFINITY) >> (threadIdx.x & 31 & ~(kLanes - 1));
    Z = fmaf(own.y, f, Z);
    for (int i0 = 0; i0 < cnt; i0 += kBatch) {
      float4 po[kBatch][kVec];
      float fi[kBatch];
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
        fi[i] = __shfl_sync(0xffffffffu, f, i0 + i, kLanes);
#pragma unroll
        for (int v = 0; v < kVec; ++v) po[i][v] = po_row[(size_t)min(s0 + i0 + i, a.splits - 1) * po_step + v];
      }
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
        const bool use = (filled >> (i0 + i)) & 1u;
#pragma unroll
        for (int v = 0; v < kVec; ++v) {
          if (!use) po[i][v] = make_float4(0.f, 0.f, 0.f, 0.f);
          acc[4 * v] = fmaf(po[i][v].x, fi[i], acc[4 * v]);
          acc[4 * v + 1] = fmaf(po[i][v].y, fi[i], acc[4 * v + 1]);
          acc[4 * v + 2] = fmaf(po[i][v].z, fi[i], acc[4 * v + 2]);
          acc[4 * v + 3] = fmaf(po[i][v].w, fi[i], acc[4 * v + 3]);
        }
      }
    }
  }
#pragma unroll
  for (int k = kLanes / 2; k > 0; k >>= 1) Z += __shfl_xor_sync(0xffffffffu, Z, k);
  float od[kChannels];
#pragma unroll
  for (int i = 0; i < kChannels; ++i) od[i] = acc[i] / Z;
  // |o|^2 over the 128 channels
  float on2 = 0.f;
#pragma unroll
  for (int v = 0; v < kVec; ++v)
    on2 += (od[4 * v] * od[4 * v] + od[4 * v + 1] * od[4 * v + 1]) + (od[4 * v + 2] * od[4 * v + 2] + od[4 * v + 3] * od[4 * v + 3]);
#pragma unroll
  for (int k = kLanes / 2; k > 0; k >>= 1) on2 += __shfl_xor_sync(0xffffffffu, on2, k);
  const size_t row = (size_t)unit * a.M + m;
  const size_t at = row * KVS_D + kChannels * lane;
  const float lse = (mstar + log2f(Z)) * 0.6931471805599453f;
  // with a supplied loss gradient the statistics need <E_q, o_q> in place of |o_q|^2
  float qconst = on2;
  if (a.e) {
    float eo = 0.f;
#pragma unroll
    for (int v = 0; v < kVec; ++v) {
      const uint2 er = *reinterpret_cast<const uint2*>(a.e + at + 4 * v);
      eo += fmaf(bf16lo(er.x), od[4 * v], bf16hi(er.x) * od[4 * v + 1]) + fmaf(bf16lo(er.y), od[4 * v + 2], bf16hi(er.y) * od[4 * v + 3]);
    }
#pragma unroll
    for (int k = kLanes / 2; k > 0; k >>= 1) eo += __shfl_xor_sync(0xffffffffu, eo, k);
    qconst = eo;
  }
  if (!mine) return;
  if (lane == 0) {
    if (a.qc2) {
      float* qc = a.qc2 + ((size_t)unit * a.M_pad + m) * 2 - (m & 1);
      qc[0] = -(mstar + log2f(Z));
      qc[2] = qconst;
    }
    if (a.lse_out) a.lse_out[row] = lse;
  }
  if (a.o_out) {
#pragma unroll
    for (int v = 0; v < kVec; ++v)
      *reinterpret_cast<float4*>(a.o_out + at + 4 * v) = make_float4(od[4 * v], od[4 * v + 1], od[4 * v + 2], od[4 * v + 3]);
  }
  struct alignas(2 * kChannels) Row { __nv_bfloat16 x[kChannels]; };
  Row hi;
#pragma unroll
  for (int i = 0; i < kChannels; ++i) hi.x[i] = __float2bfloat16_rn(od[i]);
  if (a.o_hi) {
    Row lo;
#pragma unroll
    for (int i = 0; i < kChannels; ++i) lo.x[i] = __float2bfloat16_rn(od[i] - __bfloat162float(hi.x[i]));
    *reinterpret_cast<Row*>(a.o_hi + at) = hi;
    *reinterpret_cast<Row*>(a.o_lo + at) = lo;
  }
  if (a.out_bf16) *reinterpret_cast<Row*>(a.out_bf16 + at) = hi;
}

}  // namespace

// Shared memory that the kernel does not use, so that two CTAs of the batched form fit an SM and not three.  They are
// launched while the attention still runs, onto the SMs that it leaves idle, and three to an SM slow one another
// (16 units of 80 rows: a call of the statistics 28.1 us, with two 24.6; a streaming step 65.5 and 59.7).
constexpr int kTwoPerSM = 90 * 1024;

template <int kBatch, int kLanes>
cudaError_t launch(const CombineArgs& a, const RoundTable& t, size_t smem, cudaStream_t st) {
  constexpr int kRows = kThreads / kLanes;
  const dim3 grid(((a.qc2 ? a.M_pad : a.M) + kRows - 1) / kRows, a.Hkv, t.nseq);
  return kvs_launch_chained(combine_partials<kBatch, kLanes>, grid, dim3(kThreads), smem, st, a, t);
}

cudaError_t kvs_launch_combine(const CombineArgs& a, const RoundTable& t, cudaStream_t st) {
  static KvsPerDeviceOnce configured;
  cudaError_t e = configured.run([] {
    return cudaFuncSetAttribute(combine_partials<8, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTwoPerSM);
  });
  if (e != cudaSuccess) return e;
  const long long ctas = (long long)(((a.qc2 ? a.M_pad : a.M) + 7) / 8) * a.Hkv * t.nseq;   // of eight rows
  if (ctas <= 2 * 148) return launch<8, 32>(a, t, kTwoPerSM, st);   // one wave
  if (ctas <= 4 * 148) return launch<4, 32>(a, t, 0, st);
  return launch<1, 16>(a, t, 0, st);
}
