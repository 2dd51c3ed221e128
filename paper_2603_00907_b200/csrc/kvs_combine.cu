// Combine of the attention partials that the key ranges of a query row produce.
//
// One warp per (query row, unit): the partial maxima, sums and outputs of the row's key ranges
// are merged into the row's softmax normaliser and attention output
//   o_q = sum_j alpha_qj Vsum_j / c_j,  alpha = softmax_j(scale <q, K_j> + ln c_j)   [Eq. attn_def_vec
// with merged slots].  For the observation window the kernel writes what the statistics pass needs
// (per-query constants, o as two bf16 terms); for the decode check the bf16 output.
#include "kvs_internal.h"

namespace {

// One warp per (query row, unit), eight rows per CTA; a lane owns four output channels.
constexpr int kCombineRows = 8;

// kBatch: partial outputs of a row that are requested together.  With few rows the kernel is a chain of L2
// round trips, and shorter with eight (1024 rows of 9-37 ranges: 8.5-10 -> 5.3 us); with many rows it is
// bound by bytes in flight, and the registers of a batch cost occupancy (8192 rows of 8 ranges: 9 us one by one,
// 15 us in eights; 65536 rows of 2: 24 and 75 us).  Between them four (58 registers: four CTAs to an SM): 16 units of 189 rows
// and 2 to 7 ranges 14.6 us a call, one by one 18.3, in eights 15.6; 16 units of 224 rows 83.9, 88.4 and 84.6; 32
// units of 256 rows 85.6, 84.8 and 88.9.
template <int kBatch>
__global__ void __launch_bounds__(kCombineRows * 32)
combine_partials(const CombineArgs a, const RoundTable tab) {
  kvs_pdl_launch_dependents();
  kvs_pdl_wait();
  const int seq = blockIdx.z;
  const SeqRound sr = tab.s[seq];
  if (sr.n <= 0) return;
  const int unit = sr.b * a.Hkv + blockIdx.y;
  const int m = blockIdx.x * kCombineRows + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (m >= a.M) {            // padding rows of the per-query constants: alpha = exp2(-inf) = 0
    if (lane == 0 && a.qc2 && m < a.M_pad) {
      float* qc = a.qc2 + ((size_t)unit * a.M_pad + m) * 2 - (m & 1);
      qc[0] = -INFINITY;
      qc[2] = 0.f;
    }
    return;
  }
  const size_t base = (size_t)unit * a.splits * a.M + m;
  float mstar = -INFINITY, Z = 0.f;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (kBatch == 1) {
    for (int s = 0; s < a.splits; ++s) mstar = fmaxf(mstar, a.part_ml[base + (size_t)s * a.M].x);
    for (int s = 0; s < a.splits; ++s) {
      const float2 ml = a.part_ml[base + (size_t)s * a.M];
      if (ml.x == -INFINITY) continue;
      const float f = fast_exp2(ml.x - mstar);
      Z = fmaf(ml.y, f, Z);
      const float4 po = *reinterpret_cast<const float4*>(a.part_o + (base + (size_t)s * a.M) * KVS_D + 4 * lane);
      acc.x = fmaf(po.x, f, acc.x); acc.y = fmaf(po.y, f, acc.y);
      acc.z = fmaf(po.z, f, acc.z); acc.w = fmaf(po.w, f, acc.w);
    }
  } else {
    const float2* ml = a.part_ml + base;
    const float2 first = lane < a.splits ? ml[(size_t)lane * a.M] : make_float2(-INFINITY, 0.f);
    mstar = first.x;
    for (int s = 32 + lane; s < a.splits; s += 32) mstar = fmaxf(mstar, ml[(size_t)s * a.M].x);
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) mstar = fmaxf(mstar, __shfl_xor_sync(0xffffffffu, mstar, k));
    for (int s0 = 0; s0 < a.splits; s0 += 32) {
      const int cnt = min(32, a.splits - s0);
      float2 own = first;
      if (s0 > 0) own = lane < cnt ? ml[(size_t)(s0 + lane) * a.M] : make_float2(-INFINITY, 0.f);
      const float f = own.x == -INFINITY ? 0.f : fast_exp2(own.x - mstar);
      // An empty range has left no output: what stands there is read and dropped (a condition on a load is waited for
      // before it).  One of weight 0 counts: 0 times infinity stays NaN.
      const uint32_t filled = __ballot_sync(0xffffffffu, own.x != -INFINITY);
      Z = fmaf(own.y, f, Z);
      for (int i0 = 0; i0 < cnt; i0 += kBatch) {
        float4 po[kBatch];
        float fi[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
          fi[i] = __shfl_sync(0xffffffffu, f, i0 + i);
          po[i] = *reinterpret_cast<const float4*>(a.part_o + (base + (size_t)min(s0 + i0 + i, a.splits - 1) * a.M) * KVS_D + 4 * lane);
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
          if (!((filled >> (i0 + i)) & 1u)) po[i] = make_float4(0.f, 0.f, 0.f, 0.f);
          acc.x = fmaf(po[i].x, fi[i], acc.x); acc.y = fmaf(po[i].y, fi[i], acc.y);
          acc.z = fmaf(po[i].z, fi[i], acc.z); acc.w = fmaf(po[i].w, fi[i], acc.w);
        }
      }
    }
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) Z += __shfl_xor_sync(0xffffffffu, Z, k);
  }
  const float4 od = make_float4(acc.x / Z, acc.y / Z, acc.z / Z, acc.w / Z);
  // |o|^2 over the 128 channels
  float on2 = (od.x * od.x + od.y * od.y) + (od.z * od.z + od.w * od.w);
#pragma unroll
  for (int k = 16; k > 0; k >>= 1) on2 += __shfl_xor_sync(0xffffffffu, on2, k);
  const size_t row = (size_t)unit * a.M + m;
  const float lse = (mstar + log2f(Z)) * 0.6931471805599453f;
  // with a supplied loss gradient the statistics need <E_q, o_q> in place of |o_q|^2
  float qconst = on2;
  if (a.e) {
    const uint2 er = *reinterpret_cast<const uint2*>(a.e + row * KVS_D + 4 * lane);
    float eo = fmaf(bf16lo(er.x), od.x, bf16hi(er.x) * od.y) + fmaf(bf16lo(er.y), od.z, bf16hi(er.y) * od.w);
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) eo += __shfl_xor_sync(0xffffffffu, eo, k);
    qconst = eo;
  }
  if (lane == 0) {
    if (a.qc2) {
      float* qc = a.qc2 + ((size_t)unit * a.M_pad + m) * 2 - (m & 1);
      qc[0] = -(mstar + log2f(Z));
      qc[2] = qconst;
    }
    if (a.lse_out) a.lse_out[row] = lse;
  }
  const float v[4] = {od.x, od.y, od.z, od.w};
  if (a.o_out) *reinterpret_cast<float4*>(a.o_out + row * KVS_D + 4 * lane) = od;
  if (a.o_hi) {
    __nv_bfloat16 hi[4], lo[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      hi[i] = __float2bfloat16_rn(v[i]);
      lo[i] = __float2bfloat16_rn(v[i] - __bfloat162float(hi[i]));
    }
    *reinterpret_cast<uint2*>(a.o_hi + row * KVS_D + 4 * lane) = *reinterpret_cast<const uint2*>(hi);
    *reinterpret_cast<uint2*>(a.o_lo + row * KVS_D + 4 * lane) = *reinterpret_cast<const uint2*>(lo);
  }
  if (a.out_bf16) {
    __nv_bfloat16 ob[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) ob[i] = __float2bfloat16_rn(v[i]);
    *reinterpret_cast<uint2*>(a.out_bf16 + row * KVS_D + 4 * lane) = *reinterpret_cast<const uint2*>(ob);
  }
}

}  // namespace

// Shared memory that the kernel does not use, so that two CTAs of the batched form fit an SM and not three.  They are
// launched while the attention still runs, onto the SMs that it leaves idle, and three to an SM slow one another
// (16 units of 80 rows: a call of the statistics 28.1 us, with two 24.6; a streaming step 65.5 and 59.7).
constexpr int kTwoPerSM = 90 * 1024;

cudaError_t kvs_launch_combine(const CombineArgs& a, const RoundTable& t, cudaStream_t st) {
  static KvsPerDeviceOnce configured;
  cudaError_t e = configured.run([] {
    return cudaFuncSetAttribute(combine_partials<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTwoPerSM);
  });
  if (e != cudaSuccess) return e;
  const int rows = a.qc2 ? a.M_pad : a.M;
  dim3 grid((rows + kCombineRows - 1) / kCombineRows, a.Hkv, t.nseq);
  if ((long long)grid.x * grid.y * grid.z <= 2 * 148)      // one wave
    return kvs_launch_chained(combine_partials<8>, grid, dim3(kCombineRows * 32), kTwoPerSM, st, a, t);
  if ((long long)grid.x * grid.y * grid.z <= 4 * 148)
    return kvs_launch_chained(combine_partials<4>, grid, dim3(kCombineRows * 32), 0, st, a, t);
  return kvs_launch_chained(combine_partials<1>, grid, dim3(kCombineRows * 32), 0, st, a, t);
}
