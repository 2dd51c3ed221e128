// Scores, merge weights and the exact selection of a round.
//
// A cluster of up to eight CTAs owns a (sequence, KV head) unit; a CTA owns a run of compaction tiles
// (32 candidate pairs each), a thread one pair of every 1024.  The cluster
//   1. adds the statistics kernel's partial sums of every pair in a fixed order and forms the pair's
//      score and left-key weight (for long rounds a kernel of its own does that, see below),
//   2. finds the bit pattern of the R-th smallest score by a radix select in three passes of 11, 11
//      and 10 bits (scores are non-negative floats: their bit patterns order like unsigned integers);
//      every CTA counts its own keys in shared memory and adds up the cluster's histograms,
//   3. writes the mask (ties at the cutoff are taken in index order) and, for every compaction tile,
//      the number of merged pairs that precede it.
// The keys stay in shared memory from the first step to the last.  Latency bound: barriers, L2 round trips
// and instruction fetches -- every instruction runs a few times only, so the loops are kept rolled (keys
// in registers and unrolled loops took 2.5 k cycles a pass).
// Measured, statistics' finalize + selection of a round, one CTA per unit and four passes -> this:
// 8 units of 2000 pairs 11.0 -> 7.9 us, of 16336 pairs 36.5 -> 24 us; 64 units of 2.5-32 k pairs 42 -> 27 us;
// 8 units of 65 k pairs and 24 partials a pair 73 -> 47 us.  The counts of a given mask (65 k pairs): 18 -> 7.5 us.
#include <cooperative_groups.h>

#include "kvs_internal.h"

namespace cg = cooperative_groups;

namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kKeep = 32;                  // keys of a thread held in shared memory (with more, all are read again)
constexpr int kBins = 2048;
constexpr int kMaxCluster = 8;
constexpr int kPairsPerCta = 4096, kMaskPairsPerCta = 3072;   // (see cluster_of)

// Sum of the partials of all (query block, statistics group) pairs in a fixed order, then score and
// left-key weight of candidate pair p.  Weight modes:
//   0: the sums are norms; w = (N1_l - N12) / (N1_l - 2 N12 + N1_r)                        [Eq. kstar_final]
//   1: they are the signed sums G11, G22, G12 of g_ij = E^T c_ij; w = (G11 + G12) / (G11 + 2 G12 + G22)
//                                                                            [Eq. kstar_weight_final_rewrite]
//   2: as 1 with the coupling dropped, w = G11 / (G11 + G22)                              [Eq. simplified_k]
// A denominator that is not safely positive gives 1/2; the weight is clipped to [0, 1].
__device__ __forceinline__ float finalize_pair(const StatsTcArgs& a, int unit, int off, int p) {
  const int jl = off + 2 * p;
  const int nsub = a.nqblk * KVS_STATS_GROUPS;
  const float4* p4 = a.part4 + (size_t)unit * nsub * a.pair_stride + p;
  const float* p1 = a.part1 + (size_t)unit * nsub * a.pair_stride + p;
  float Al = 0.f, Ar = 0.f, N1l = 0.f, N1r = 0.f, N12 = 0.f;
  for (int sb = 0; sb < nsub; sb += KVS_STATS_GROUPS) {
    float4 v[KVS_STATS_GROUPS];
    float x[KVS_STATS_GROUPS];
#pragma unroll
    for (int i = 0; i < KVS_STATS_GROUPS; ++i) {
      v[i] = p4[(size_t)(sb + i) * a.pair_stride];
      x[i] = p1[(size_t)(sb + i) * a.pair_stride];
    }
#pragma unroll
    for (int i = 0; i < KVS_STATS_GROUPS; ++i) { Al += v[i].x; Ar += v[i].y; N1l += v[i].z; N1r += v[i].w; N12 += x[i]; }
  }
  const float cosv = a.pair_norms[(size_t)unit * a.norm_stride + p].w;
  const float mass = Al + Ar;
  const float score = (a.score_mode == 0) ? mass * fmaxf(0.f, 1.f - cosv) : mass;
  float w = 0.5f;
  if (a.weight_mode == 0) {
    const float D = N1l - 2.f * N12 + N1r;
    if (D > 1e-6f * (N1l + N1r) && D < INFINITY) w = fminf(1.f, fmaxf(0.f, (N1l - N12) / D));
  } else {
    const float g12 = (a.weight_mode == 2) ? 0.f : N12;
    const float gamma = N1l + 2.f * g12 + N1r;
    if (gamma > 1e-6f * (fabsf(N1l) + fabsf(N1r)) && gamma < INFINITY) w = fminf(1.f, fmaxf(0.f, (N1l + g12) / gamma));
  }
  const size_t pi = (size_t)unit * a.pair_stride + p;
  a.score[pi] = fabsf(score);
  a.w[pi] = w;
  if (a.N12) a.N12[pi] = N12;
  if (a.cosv) a.cosv[pi] = cosv;
  if (a.A) { a.A[(size_t)unit * a.n_max + jl] = Al; a.A[(size_t)unit * a.n_max + jl + 1] = Ar; }
  if (a.N1) { a.N1[(size_t)unit * a.n_max + jl] = N1l; a.N1[(size_t)unit * a.n_max + jl + 1] = N1r; }
  return fabsf(score);
}

// Exclusive prefix of `v` over the threads of the CTA (one barrier; `s_warp` is free again after the next one).
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  uint32_t w = s_warp[lane];                               // (32 warps, 32 lanes)
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, w, o);
    if (lane >= o) w += t;
  }
  const uint32_t before = warp ? __shfl_sync(0xffffffffu, w, warp - 1) : 0u;
  return before + inc - v;
}

// Step 1 alone, over the whole GPU: one thread per pair.
__global__ void __launch_bounds__(256)
finalize_kernel(const StatsTcArgs a, const RoundTable tab) {
  kvs_pdl_launch_dependents();
  kvs_pdl_wait();
  const SeqRound sr = tab.s[blockIdx.z];
  const int p = blockIdx.x * 256 + threadIdx.x;
  if (sr.n <= 0 || p >= sr.P) return;
  finalize_pair(a, sr.b * a.Hkv + blockIdx.y, tab.off, p);
}

// kFused: step 1 too; kScores: the scores are in memory; kMask: the mask is an input (kvs_compact) and only
// the counts of step 3 are formed.
enum { kFused = 0, kScores = 1, kMask = 2 };
template <int kMode>
__global__ void __launch_bounds__(kThreads, 2)
select_kernel(const StatsTcArgs sa, const SelectArgs a, const RoundTable tab) {
  constexpr bool kFromMask = kMode == kMask;
  extern __shared__ uint32_t s_key[];
  __shared__ alignas(8) uint32_t s_hist[3][kBins];       // (read as pairs of bins)
  __shared__ uint32_t s_warp[2][kWarps], s_digit, s_k, s_total[2], s_cnt[2][kWarps];
  kvs_pdl_launch_dependents();
  cg::cluster_group cluster = cg::this_cluster();
  const int ctas = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < 2) s_total[tid] = 0;
  if (!kFromMask)
    for (int i = tid; i < 3 * kBins; i += kThreads) (&s_hist[0][0])[i] = 0;
  kvs_pdl_wait();
  {
    const uint32_t cta = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x, all = gridDim.x * gridDim.y * gridDim.z;
    for (uint32_t i = cta * kThreads + tid; i < a.zero_bytes / 16; i += all * kThreads) a.zero[i] = make_uint4(0, 0, 0, 0);
  }
  const SeqRound sr = tab.s[blockIdx.z];
  const int n = sr.n;
  if (n <= 0) return;                                      // (the whole cluster)
  const int unit = sr.b * a.Hkv + blockIdx.y;
  const int P = sr.P;
  // this CTA's compaction tiles and pairs
  const int ntiles = max(0, n - tab.off + KVS_CTILE - 1) / KVS_CTILE;
  const int per_cta = (ntiles + ctas - 1) / ctas;
  const int t0 = min(ntiles, rank * per_cta), t1 = min(ntiles, t0 + per_cta);
  const int steps = (t1 - t0 + kWarps - 1) / kWarps;       // of 32 tiles = 1024 pairs
  const int p_end = min(P, 32 * t1);
  const int p_first = 32 * t0 + tid;
  uint8_t* mask = a.mask + (size_t)unit * a.pair_stride;
  const uint32_t* score = reinterpret_cast<const uint32_t*>(sa.score) + (size_t)unit * a.pair_stride;

  if (!kFromMask) {
#pragma unroll 1
    for (int u = 0, p = p_first; p < p_end; ++u, p += kThreads) {
      const uint32_t x = kMode == kFused ? __float_as_uint(finalize_pair(sa, unit, tab.off, p)) : score[p];
      if (steps <= kKeep) s_key[u * kThreads + tid] = x;
    }
  }
  // the keys of this CTA (every thread reads only what it has written itself)
  const uint32_t* keys = steps <= kKeep ? s_key + tid : score + p_first;
  auto key_of = [&](int u, int p) -> uint32_t {
    if (p >= p_end) return 0u;
    return kFromMask ? (uint32_t)mask[p] : keys[(size_t)u * kThreads];
  };
  auto cluster_barrier = [&] { if (ctas > 1) cluster.sync(); else __syncthreads(); };

  // ---- cutoff: bit pattern of the R-th smallest score; k of its ties are taken
  uint32_t cutoff = 0, k = kFromMask ? 0u : (uint32_t)sr.R;
  __syncthreads();
  if (!kFromMask) {
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
      const int shift = pass == 0 ? 21 : pass == 1 ? 10 : 0;
      const int bits = pass == 2 ? 10 : 11;
#pragma unroll 1
      for (int u = 0, p = p_first; p < p_end; ++u, p += kThreads) {
        const uint32_t v = key_of(u, p);
        if (pass == 0 || ((v ^ cutoff) >> (shift + bits)) == 0) atomicAdd(&s_hist[pass][(v >> shift) & ((1u << bits) - 1u)], 1u);
      }
      cluster_barrier();
      uint2 h = make_uint2(0, 0);
#pragma unroll 1
      for (int r = 0; r < ctas; ++r) {
        const uint2 x = *cluster.map_shared_rank(reinterpret_cast<uint2*>(&s_hist[pass][2 * tid]), r);
        h.x += x.x; h.y += x.y;
      }
      const uint32_t before = block_scan(h.x + h.y, s_warp[pass & 1]);
      if (before < k && k <= before + h.x) { s_digit = 2 * tid; s_k = k - before; }
      if (before + h.x < k && k <= before + h.x + h.y) { s_digit = 2 * tid + 1; s_k = k - before - h.x; }
      __syncthreads();
      cutoff |= s_digit << shift;
      k = s_k;
    }
  }
  // ---- pairs below the cutoff and at it, in this CTA and in the CTAs before it
  uint32_t below = 0, at = 0;
#pragma unroll 1
  for (int u = 0, p = p_first; p < p_end; ++u, p += kThreads) {
    const uint32_t v = key_of(u, p);
    below += (kFromMask ? v != 0 : v < cutoff) ? 1u : 0u;
    at += (!kFromMask && v == cutoff) ? 1u : 0u;
  }
  below = __reduce_add_sync(0xffffffffu, below);
  at = __reduce_add_sync(0xffffffffu, at);
  if (lane == 0 && below) atomicAdd(&s_total[0], below);
  if (lane == 0 && at) atomicAdd(&s_total[1], at);
  cluster_barrier();
  below = at = 0;
  for (int r = 0; r < rank; ++r) {
    below += *cluster.map_shared_rank(&s_total[0], r);
    at += *cluster.map_shared_rank(&s_total[1], r);
  }
  // ---- mask and counts in front of every tile, 32 tiles (one per warp) a step.  The first k ties are taken.
  int32_t* tp = a.tile_prefix + (size_t)unit * a.tile_stride;
#pragma unroll 1
  for (int u = 0; u < steps; ++u) {
    const int p = p_first + u * kThreads;
    const uint32_t v = key_of(u, p);
    const bool lt = p < p_end && (kFromMask ? v != 0 : v < cutoff);
    const bool eq = !kFromMask && p < p_end && v == cutoff;
    const uint32_t bl = __ballot_sync(0xffffffffu, lt), be = __ballot_sync(0xffffffffu, eq);
    uint32_t* cnt = s_cnt[u & 1];
    if (lane == 0) cnt[warp] = __popc(bl) | (__popc(be) << 16);
    __syncthreads();
    uint32_t c = cnt[lane];                                // (32 warps, 32 lanes; the sums stay below 2^16)
    const uint32_t own = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, c, o);
      if (lane >= o) c += t;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, c, 31), ex = __shfl_sync(0xffffffffu, c - own, warp);
    const uint32_t tie_before = at + (ex >> 16);
    if (!kFromMask && p < p_end) mask[p] = (lt || (eq && tie_before + __popc(be & ((1u << lane) - 1u)) < k)) ? 1 : 0;
    const int tile = t0 + u * kWarps + warp;
    if (lane == 0 && tile < t1) tp[tile] = (int32_t)(below + (ex & 0xffffu) + min(k, tie_before));
    below += total & 0xffffu;
    at += total >> 16;
  }
  if (ctas > 1) cluster.sync();                            // no CTA leaves while its shared memory is read
}

int most_pairs(const RoundTable& t) {
  int pmax = 0;
  for (int i = 0; i < t.nseq; ++i) pmax = pmax > t.s[i].P ? pmax : t.s[i].P;
  return pmax;
}

// CTAs per unit: one for every 4096 pairs while they all fit the GPU (two per SM).  A cluster's barriers cost about
// 1.5 us each: 8 units of 16336 pairs 17 us with four CTAs, 28 with eight; 256 units of 16336 pairs 32 us with
// one, 85 with several waves of clusters of four.  The counts of a given mask have one such barrier and take a CTA for
// 3072 pairs: a compaction of 4 units of 7200 pairs 22.1 us, with half as many 24.0; of 8 units of 16336 63.2 and 64.4;
// but of 32 units of 2180 74.4 with two CTAs and 70.8 with one.
int cluster_of(const RoundTable& t, int Hkv, int pairs_per_cta) {
  const int pmax = most_pairs(t);
  int c = 1;
  while (c < kMaxCluster && c * pairs_per_cta < pmax && (long long)c * 2 * Hkv * t.nseq <= 2 * 148) c *= 2;
  return c;
}

constexpr int kSpreadSmem = 118 * 1024;
static_assert(kSpreadSmem <= kKeep * kThreads * (int)sizeof(uint32_t), "the kernel is configured for its keys");
template <int kMode>
cudaError_t launch_select(const StatsTcArgs& sa, const SelectArgs& a, const RoundTable& t, cudaStream_t st) {
  static KvsPerDeviceOnce configured;
  cudaError_t e = configured.run([] {
    return cudaFuncSetAttribute(select_kernel<kMode>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kKeep * kThreads * (int)sizeof(uint32_t));
  });
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  const int c = cluster_of(t, a.Hkv, kMode == kMask ? kMaskPairsPerCta : kPairsPerCta);
  cfg.gridDim = dim3((unsigned)c, (unsigned)a.Hkv, (unsigned)t.nseq);
  cfg.blockDim = dim3(kThreads);
  if (kMode != kMask) {
    int nmax = 0;
    for (int i = 0; i < t.nseq; ++i) nmax = nmax > t.s[i].n ? nmax : t.s[i].n;
    const int ntiles = (nmax - t.off + KVS_CTILE - 1) / KVS_CTILE;
    const int steps = ((ntiles + c - 1) / c + kWarps - 1) / kWarps;
    cfg.dynamicSmemBytes = (size_t)(steps <= kKeep ? steps : kKeep) * kThreads * sizeof(uint32_t);   // (shorter units keep theirs)
  }
  // The statistics kernel fills every SM when it walks equal shares: the selection's CTAs then all start on the
  // few SMs that are done first, where they slow one another (8 units of 1200 pairs: 16 us against 10.8).
  // Shared memory for one CTA per SM spreads them.
  if (kMode != kMask && sa.splits == 0 && (long long)c * a.Hkv * t.nseq <= 148 && cfg.dynamicSmemBytes < (size_t)kSpreadSmem)
    cfg.dynamicSmemBytes = kSpreadSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)c;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, select_kernel<kMode>, sa, a, t);
}

// Whether the selection kernel adds the partials itself: where they are few (at most two query blocks), and
//   * a unit has up to 1024 pairs: 8 units of 350 30.3 us a call against 31.1 with a kernel of its own, 32 of 700 40.4 and 43.8;
//   * there are up to 16 units of up to 3072 pairs, or up to 44000 pairs in all: 16 of 2000 42.5 us and 46.3, 8 of 3000 42.3
//     and 44.5, 24 of 1760 51.1 and 55.4;
//   * the units are enough for the GPU: 128 of 2000 175 us and 186.
// Between them its few CTAs are slow readers: 24 units of 3000 pairs 74 us against 64, 32 of 2000 67 and 61, 64 of 4000
// 195 and 183, 16 of 4000 63 and 61.
bool fused_finalize(const StatsTcArgs& sa, const SelectArgs& a, int units, int pmax) {
  if (!a.select || sa.nqblk > 2 || pmax > 4096) return false;
  return pmax <= 1024 || units >= 128 || (pmax <= 3072 && (units <= 16 || pmax * units <= 44000));
}

}  // namespace

cudaError_t kvs_launch_finalize_select(const StatsTcArgs& sa, const SelectArgs& a, const RoundTable& t, cudaStream_t st,
                                       int* kernels) {
  *kernels = 1;
  const int pmax = most_pairs(t);
  if (pmax <= 0) return cudaSuccess;
  if (fused_finalize(sa, a, a.Hkv * t.nseq, pmax)) return launch_select<kFused>(sa, a, t, st);
  cudaError_t e = kvs_launch_chained(finalize_kernel, dim3((pmax + 255) / 256, a.Hkv, t.nseq), dim3(256), 0, st, sa, t);
  if (e != cudaSuccess || !a.select) return e;
  *kernels = 2;
  return launch_select<kScores>(sa, a, t, st);
}

cudaError_t kvs_launch_mask_prefix(const SelectArgs& a, const RoundTable& t, cudaStream_t st) {
  return launch_select<kMask>(StatsTcArgs{}, a, t, st);
}
