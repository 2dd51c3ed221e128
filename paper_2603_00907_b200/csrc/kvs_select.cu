// Scores, merge weights and the exact selection of a round.
//
// A cluster of up to eight CTAs owns a (sequence, KV head) unit; a CTA owns a run of compaction tiles
// (32 candidate pairs each), a warp a run of these, a lane one pair of each.  The cluster
//   1. adds the statistics kernel's partial sums of every pair in a fixed order and forms the pair's
//      score and left-key weight (for long rounds a kernel of its own does that, see below),
//   2. finds the bit pattern of the R-th smallest score (scores are non-negative floats: their bit patterns order
//      like unsigned integers).  A pass counts the keys of an interval in 4096 bins and goes on with the bin
//      that holds the R-th; two passes are the rule, since it ends when a bin is taken as a whole,
//   3. writes the mask (ties at the cutoff are taken in index order) and, for every compaction tile,
//      the number of merged pairs that precede it.
// A warp owns consecutive tiles, so that the counts in front of a tile need one barrier a launch.
// The keys stay in shared memory from the first step to the last.  Latency bound: barriers (of a cluster 1.1 k cycles
// each), L2 round trips and issue slots, of which an instruction of all 1024 threads takes eight on every scheduler.
// Measured, clock64 from the wait for the kernel before to the end, three passes of 11, 11 and 10 bits with all counts
// read from the other CTAs and a barrier for every 1024 pairs -> this: 8 units of 2000 pairs 14.7 -> 11.0 k cycles, of
// 4096 16.2 -> 10.4, of 16336 23.9 -> 13.7, of 65 k 41.8 -> 20.4 k.  With the finalize kernel, us by events: 8 units of 16336
// pairs 28.0 -> 17.9, 13 rounds of 8 units from 65 k pairs on 557 -> 428.
// (Listing the keys of the first pass's bin and ranking them by comparison in place of the second pass: 140 keys
// 3.7 k cycles, 480 keys 18 k.)
#include <cooperative_groups.h>

#include "kvs_internal.h"

namespace cg = cooperative_groups;

namespace {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kKeep = 32;                  // keys of a thread held in shared memory (with more, all are read again)
constexpr int kBinBits = 12, kBins = 1 << kBinBits;   // of a pass
static_assert(kBins == 4 * kThreads, "a thread sums four bins");
constexpr int kMaxCluster = 8;
constexpr int kPairsPerCta = 4096, kMaskPairsPerCta = 3072;   // (see cluster_of)

// Sum of the partials of all (query block, statistics group) pairs in a fixed order, then score and
// left-key weight of candidate pair p.  Weight modes:
//   0: the sums are norms; w = (N1_l - N12) / (N1_l - 2 N12 + N1_r)                        [Eq. kstar_final]
//   1: they are the signed sums G11, G22, G12 of g_ij = E^T c_ij; w = (G11 + G12) / (G11 + 2 G12 + G22)
//                                                                            [Eq. kstar_weight_final_rewrite]
//   2: as 1 with the coupling dropped, w = G11 / (G11 + G22)                              [Eq. simplified_k]
// A denominator that is not safely positive gives 1/2; the weight is clipped to [0, 1].
struct PairSums { float Al, Ar, N1l, N1r, N12, cosv; };
__device__ __forceinline__ PairSums pair_sums(const StatsTcArgs& a, int unit, int p) {
  const int nsub = a.nqblk * KVS_STATS_GROUPS;
  const float4* p4 = a.part4 + (size_t)unit * nsub * a.pair_stride + p;
  const float* p1 = a.part1 + (size_t)unit * nsub * a.pair_stride + p;
  PairSums s = {0.f, 0.f, 0.f, 0.f, 0.f, a.pair_norms[(size_t)unit * a.norm_stride + p].w};
  for (int sb = 0; sb < nsub; sb += KVS_STATS_GROUPS) {
    float4 v[KVS_STATS_GROUPS];
    float x[KVS_STATS_GROUPS];
#pragma unroll
    for (int i = 0; i < KVS_STATS_GROUPS; ++i) {
      v[i] = p4[(size_t)(sb + i) * a.pair_stride];
      x[i] = p1[(size_t)(sb + i) * a.pair_stride];
    }
#pragma unroll
    for (int i = 0; i < KVS_STATS_GROUPS; ++i) { s.Al += v[i].x; s.Ar += v[i].y; s.N1l += v[i].z; s.N1r += v[i].w; s.N12 += x[i]; }
  }
  return s;
}
__device__ __forceinline__ float finish_pair(const StatsTcArgs& a, int unit, int off, int p, const PairSums& s) {
  const int jl = off + 2 * p;
  const float mass = s.Al + s.Ar;
  const float score = (a.score_mode == 0) ? mass * fmaxf(0.f, 1.f - s.cosv) : mass;
  float w = 0.5f;
  if (a.weight_mode == 0) {
    const float D = s.N1l - 2.f * s.N12 + s.N1r;
    if (D > 1e-6f * (s.N1l + s.N1r) && D < INFINITY) w = fminf(1.f, fmaxf(0.f, (s.N1l - s.N12) / D));
  } else {
    const float g12 = (a.weight_mode == 2) ? 0.f : s.N12;
    const float gamma = s.N1l + 2.f * g12 + s.N1r;
    if (gamma > 1e-6f * (fabsf(s.N1l) + fabsf(s.N1r)) && gamma < INFINITY) w = fminf(1.f, fmaxf(0.f, (s.N1l + g12) / gamma));
  }
  const size_t pi = (size_t)unit * a.pair_stride + p;
  a.score[pi] = fabsf(score);
  a.w[pi] = w;
  if (a.N12) a.N12[pi] = s.N12;
  if (a.cosv) a.cosv[pi] = s.cosv;
  if (a.A) { a.A[(size_t)unit * a.n_max + jl] = s.Al; a.A[(size_t)unit * a.n_max + jl + 1] = s.Ar; }
  if (a.N1) { a.N1[(size_t)unit * a.n_max + jl] = s.N1l; a.N1[(size_t)unit * a.n_max + jl + 1] = s.N1r; }
  return fabsf(score);
}

// Inclusive prefix over the lanes of the warp.
__device__ __forceinline__ uint32_t warp_scan(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Step 1 alone, over the whole GPU: one thread per pair.
__global__ void __launch_bounds__(256)
finalize_kernel(const StatsTcArgs a, const RoundTable tab) {
  kvs_pdl_launch_dependents();
  kvs_pdl_wait();
  const SeqRound sr = tab.s[blockIdx.z];
  const int p = blockIdx.x * 256 + threadIdx.x;
  if (sr.n <= 0 || p >= sr.P) return;
  const int unit = sr.b * a.Hkv + blockIdx.y;
  finish_pair(a, unit, tab.off, p, pair_sums(a, unit, p));
}

// A key: the bits of a score, which is not negative (nor has a NaN its sign here: every key lies in the first interval).
constexpr uint32_t kKeyBits = 0x7fffffffu;
// Passes until the interval is one pattern: the widest bin of the first pass has 2^30 of them, a later pass divides by 2^12.
constexpr int kPasses = 4;
// The digit of the first pass: 64 bins to an octave of the score from 2^-56 to 2^8; what lies outside joins the first
// or the last bin.  (It grows with the score, and the bins are so narrow that few scores share the cutoff's.)
constexpr int kFirstBin = (127 - 56) << 6;
__device__ __forceinline__ int first_digit(uint32_t v) { return min(max((int)(v >> 17) - kFirstBin, 0), kBins - 1); }

// kFused: step 1 too; kScores: the scores are in memory; kMask: the mask is an input (kvs_compact) and only
// the counts of step 3 are formed.  kFusedFew: as kFused, with the registers of a whole SM to a CTA and two pairs a thread in flight
// (8 units of 2000 pairs: the first step 6700 -> 4700 cycles, most of which the partials' 150 KB take to get to one SM).
// kCluster: more than one CTA to a unit; with the scores in memory one CTA to an SM, too: at the 32 registers of two, the
// passes spilled (8 units of 16336 pairs: 21.7 k cycles against 13.7 k).
enum { kFused = 0, kScores = 1, kMask = 2, kFusedFew = 3 };
template <int kMode, bool kCluster>
__global__ void __launch_bounds__(kThreads, kMode == kFusedFew || (kMode == kScores && kCluster) ? 1 : 2)
select_kernel(const StatsTcArgs sa, const SelectArgs a, const RoundTable tab) {
  constexpr bool kFromMask = kMode == kMask;
  extern __shared__ uint32_t s_key[];
  // two passes' counts in turn: a CTA still reads those of one pass when another one counts for the next
  __shared__ alignas(16) uint32_t s_hist[kFromMask ? 1 : 2][kFromMask ? 4 : kBins];
  __shared__ uint32_t s_coarse[2][kWarps], s_pick[3], s_below[kWarps], s_at[kWarps];
  kvs_pdl_launch_dependents();
  cg::cluster_group cluster = cg::this_cluster();
  const int ctas = kCluster ? (int)cluster.num_blocks() : 1, rank = kCluster ? (int)cluster.block_rank() : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (!kFromMask)
    for (int i = tid; i < 2 * kBins; i += kThreads) (&s_hist[0][0])[i] = 0;
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
  // this CTA's compaction tiles, and this warp's: `steps` of them, one pair of each to a lane
  const int ntiles = max(0, n - tab.off + KVS_CTILE - 1) / KVS_CTILE;
  const int per_cta = (ntiles + ctas - 1) / ctas;
  const int t0 = min(ntiles, rank * per_cta), t1 = min(ntiles, t0 + per_cta);
  const int steps = (t1 - t0 + kWarps - 1) / kWarps;
  const int tile0 = t0 + warp * steps;
  const int p_end = min(P, 32 * t1);
  const int p_first = 32 * tile0 + lane;
  uint8_t* mask = a.mask + (size_t)unit * a.pair_stride;
  const uint32_t* score = reinterpret_cast<const uint32_t*>(sa.score) + (size_t)unit * a.pair_stride;

  if (kMode == kFused) {
#pragma unroll 1
    for (int u = 0, p = p_first; u < steps && p < p_end; ++u, p += 32) {
      const float x = finish_pair(sa, unit, tab.off, p, pair_sums(sa, unit, p));
      if (steps <= kKeep) s_key[u * kThreads + tid] = __float_as_uint(x) & kKeyBits;
    }
  } else if (kMode == kFusedFew) {
#pragma unroll 1
    for (int u = 0, p = p_first; u < steps && p < p_end; u += 2, p += 64) {
      const bool two = u + 1 < steps && p + 32 < p_end;
      const PairSums x = pair_sums(sa, unit, p), y = pair_sums(sa, unit, two ? p + 32 : p);
      const float sx = finish_pair(sa, unit, tab.off, p, x);
      const float sy = two ? finish_pair(sa, unit, tab.off, p + 32, y) : 0.f;
      if (steps <= kKeep) {
        s_key[u * kThreads + tid] = __float_as_uint(sx) & kKeyBits;
        if (two) s_key[(u + 1) * kThreads + tid] = __float_as_uint(sy) & kKeyBits;
      }
    }
  } else if (kMode == kScores && steps <= kKeep) {
#pragma unroll 4
    for (int u = 0; u < steps; ++u) s_key[u * kThreads + tid] = p_first + 32 * u < p_end ? score[p_first + 32 * u] & kKeyBits : 0u;
  }
  // (pairs are at most 3072 in the fused modes, but a unit with a long protected suffix has more tiles, and more steps than
  // are kept: then the scores just written are read again)
  // the key of a step (every thread reads only what it has written itself)
  auto key_of = [&](int u) -> uint32_t {
    const int p = p_first + 32 * u;
    if (p >= p_end) return 0u;
    return kFromMask ? (uint32_t)mask[p] : steps <= kKeep ? s_key[u * kThreads + tid] : score[p] & kKeyBits;
  };
  auto cluster_barrier = [&] { if (kCluster) cluster.sync(); else __syncthreads(); };
  auto of_rank = [&](auto* x, int r) { return kCluster ? *cluster.map_shared_rank(x, r) : *x; };

  // ---- cutoff: bit pattern of the R-th smallest score; k of its ties are taken.  Every pass cuts the interval
  //      [lo, lo + width) that holds it into up to 4096 bins, until the interval is one pattern or is taken as a whole.
  uint32_t cutoff = 0, k = kFromMask ? 0u : (uint32_t)sr.R;
  if (!kFromMask) {
    uint32_t lo = 0, width = kKeyBits + 1u;
    __syncthreads();
#pragma unroll 1
    for (int pass = 0; pass < kPasses; ++pass) {
      uint32_t* hist = s_hist[pass & 1];
      if (pass >= 2) {
        for (int i = tid; i < kBins; i += kThreads) hist[i] = 0;
        __syncthreads();
      }
      const int shift = max(0, 32 - __clz((int)(width - 1)) - kBinBits);
#pragma unroll 2
      for (int u = 0; u < steps; ++u) {
        const uint32_t v = key_of(u);
        if (p_first + 32 * u < p_end && v - lo < width) atomicAdd(&hist[pass == 0 ? (uint32_t)first_digit(v) : (v - lo) >> shift], 1u);
      }
      __syncthreads();
      // The 128 bins that hold the k-th key are found from the sums of 128, its bin from their counts: little is read of the
      // other CTAs' shared memory (all counts of three CTAs: 1400 cycles, of seven 2700), and one warp does it (all of
      // them, redundantly, took 1000 cycles a pass more: with 1024 threads an instruction is eight issue slots).
      uint32_t* coarse = s_coarse[pass & 1];
      const uint4 mine = reinterpret_cast<const uint4*>(s_hist[pass & 1])[tid];
      const uint32_t of_mine = __reduce_add_sync(0xffffffffu, mine.x + mine.y + mine.z + mine.w);
      if (lane == 0) coarse[warp] = of_mine;
      cluster_barrier();
      if (warp == 0) {
        uint32_t sum = 0;
#pragma unroll 4
        for (int r = 0; r < ctas; ++r) sum += of_rank(&coarse[lane], r);
        const uint32_t upto = warp_scan(sum);
        const int hit = (__ffs((int)__ballot_sync(0xffffffffu, upto >= k)) - 1) & 31;
        uint32_t before = __shfl_sync(0xffffffffu, upto - sum, hit);
        uint32_t h[4] = {0, 0, 0, 0};
#pragma unroll 4
        for (int r = 0; r < ctas; ++r) {
          const uint4 x = of_rank(reinterpret_cast<uint4*>(s_hist[pass & 1]) + 32 * hit + lane, r);
          h[0] += x.x; h[1] += x.y; h[2] += x.z; h[3] += x.w;
        }
        const uint32_t own = (h[0] + h[1]) + (h[2] + h[3]);
        before += warp_scan(own) - own;
        bool found = false;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (before < k && k <= before + h[i]) {
            s_pick[0] = 4 * (32 * hit + lane) + i; s_pick[1] = k - before; s_pick[2] = h[i];
            found = true;
          }
          before += h[i];
        }
        if (!__any_sync(0xffffffffu, found) && lane == 0) s_pick[2] = 0;
      }
      __syncthreads();
      const uint32_t bin = s_pick[0], in_bin = s_pick[2];
      if (in_bin == 0) {                                   // no bin holds it: never, as long as 1 <= R <= P
        if (tid == 0 && sa.status_dev) atomicExch(sa.status_dev, (int)KVS_ERR_CUDA);
        k = 0;
        break;
      }
      k = s_pick[1];
      if (pass == 0) {
        lo = bin == 0 ? 0u : (bin + kFirstBin) << 17;
        width = (bin == kBins - 1 ? kKeyBits + 1u : (bin + kFirstBin + 1) << 17) - lo;
      } else {
        width = min(1u << shift, width - (bin << shift));
        lo += bin << shift;
      }
      if (in_bin == k) { cutoff = lo + width; k = 0; break; }
      if (width == 1) { cutoff = lo; break; }
    }
  }
  // ---- pairs below the cutoff and at it, in this warp ...
  uint32_t below = 0, at = 0, kept = 0;
#pragma unroll 4
  for (int u = 0; u < steps; ++u) {
    const uint32_t v = key_of(u);
    const bool in = p_first + 32 * u < p_end;
    const uint32_t c = __popc(__ballot_sync(0xffffffffu, in && (kFromMask ? v != 0 : v < cutoff)));
    below += c;
    if (kFromMask && lane == (u & 31)) kept = c;
    if (!kFromMask && k != 0) at += __popc(__ballot_sync(0xffffffffu, in && v == cutoff));
  }
  if (lane == 0) { s_below[warp] = below; s_at[warp] = at; }
  cluster_barrier();
  // ... and in front of it
  below = lane < warp ? s_below[lane] : 0u;
  at = lane < warp ? s_at[lane] : 0u;
  for (int r = 0; r < rank; ++r) {
    below += of_rank(&s_below[lane], r);
    if (!kFromMask) at += of_rank(&s_at[lane], r);
  }
  below = __reduce_add_sync(0xffffffffu, below);
  if (!kFromMask) at = __reduce_add_sync(0xffffffffu, at);
  // ---- mask and counts in front of every tile.  The first k ties are taken.
  int32_t* tp = a.tile_prefix + (size_t)unit * a.tile_stride;
  if (kFromMask && steps <= 32) {
    const uint32_t upto = warp_scan(kept);
    if (lane < steps && tile0 + lane < t1) tp[tile0 + lane] = (int32_t)(below + upto - kept);
  } else {
#pragma unroll 2
    for (int u = 0; u < steps; ++u) {
      const int p = p_first + 32 * u;
      const uint32_t v = key_of(u);
      const bool in = p < p_end;
      const bool lt = in && (kFromMask ? v != 0 : v < cutoff);
      bool taken = lt;
      if (lane == 0 && tile0 + u < t1) tp[tile0 + u] = (int32_t)(below + min(k, at));
      below += __popc(__ballot_sync(0xffffffffu, lt));
      if (!kFromMask && k != 0) {                          // (mostly the interval was taken as a whole, and there are no ties)
        const uint32_t be = __ballot_sync(0xffffffffu, in && v == cutoff);
        taken = lt || (in && v == cutoff && at + __popc(be & ((1u << lane) - 1u)) < k);
        at += __popc(be);
      }
      if (!kFromMask && in) mask[p] = taken ? 1 : 0;
    }
  }
  if (kCluster) cluster.sync();                            // no CTA leaves while its shared memory is read
}

int most_pairs(const RoundTable& t) {
  int pmax = 0;
  for (int i = 0; i < t.nseq; ++i) pmax = pmax > t.s[i].P ? pmax : t.s[i].P;
  return pmax;
}

// CTAs per unit: one for every 4096 pairs while they all fit the GPU, one per SM (6144 and 8192: a call of the statistics of 8
// units of 16336 pairs 132.0 and 134.0 us, with 4096 132.3; nine rounds of 8 units from 16 k pairs on 148, 152 and
// 144 us in the selections; 256 units of 16336 pairs 32 us with one, 85 with several waves of clusters of
// four).  The counts of a given mask need few registers: two per SM, a CTA for
// 3072 pairs: a compaction of 4 units of 7200 pairs 22.1 us, with half as many 24.0; of 8 units of 16336 63.2 and 64.4;
// but of 32 units of 2180 74.4 with two CTAs and 70.8 with one.
int cluster_of(const RoundTable& t, int Hkv, int pairs_per_cta, int fit) {
  const int pmax = most_pairs(t);
  int c = 1;
  while (c < kMaxCluster && c * pairs_per_cta < pmax && (long long)c * 2 * Hkv * t.nseq <= fit) c *= 2;
  return c;
}

constexpr int kSpreadSmem = 118 * 1024;
static_assert(kSpreadSmem <= kKeep * kThreads * (int)sizeof(uint32_t), "the kernel is configured for its keys");
template <int kMode, bool kCluster>
cudaError_t launch_select(const StatsTcArgs& sa, const SelectArgs& a, const RoundTable& t, int c, cudaStream_t st) {
  static KvsPerDeviceOnce configured;
  cudaError_t e = configured.run([] {
    return cudaFuncSetAttribute(select_kernel<kMode, kCluster>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kKeep * kThreads * (int)sizeof(uint32_t));
  });
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
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
  cfg.numAttrs = kCluster ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, select_kernel<kMode, kCluster>, sa, a, t);
}

// Whether the selection kernel adds the partials itself: where they are few (at most two query blocks), and a unit has up to
// 1536 pairs, or up to 3072 with up to 16 units.  Its few CTAs are slow readers of more.  Us a call of the statistics with a
// kernel of its own for the partials and without, 64 rows: 8 units of 700 pairs 28.5 and 24.5, of 2000 30.4 and 27.9, of 3000 34.6 and 34.8; 16 of
// 3000 43.5 and 40.8; 24 of 1500 36.7 and 34.3, of 3000 49.4 and 50.2, of 4000 60.4 and 62.7; 32 of 1500 41.7 and 38.9, of 2000 46.5 and
// 45.6; 64 of 1500 67.2 and 65.5, of 4000 137 and 139; 128 of 1500 112 and 110; 256 of 1500 208.9 and 208.2, of 3000 371 and 387; 256 rows: 16
// of 3000 68.6 and 67.1; 32 of 1500 69.4 and 65.7, of 3000 110 and 112; 128 of 1500 217 and 215, of 2000 264 and 274; 256 of 2000 506 and 540.
bool fused_finalize(const StatsTcArgs& sa, const SelectArgs& a, int units, int pmax) {
  if (!a.select || sa.nqblk > 2) return false;
  return pmax <= 1536 || (pmax <= 3072 && units <= 16);
}

}  // namespace

cudaError_t kvs_launch_finalize_select(const StatsTcArgs& sa, const SelectArgs& a, const RoundTable& t, cudaStream_t st,
                                       int* kernels) {
  *kernels = 1;
  const int pmax = most_pairs(t);
  if (pmax <= 0) return cudaSuccess;
  const int units = a.Hkv * t.nseq;
  if (fused_finalize(sa, a, units, pmax))                  // (so few pairs a unit: one CTA)
    return units <= 148 ? launch_select<kFusedFew, false>(sa, a, t, 1, st) : launch_select<kFused, false>(sa, a, t, 1, st);
  cudaError_t e = kvs_launch_chained(finalize_kernel, dim3((pmax + 255) / 256, a.Hkv, t.nseq), dim3(256), 0, st, sa, t);
  if (e != cudaSuccess || !a.select) return e;
  *kernels = 2;
  const int c = cluster_of(t, a.Hkv, kPairsPerCta, 148);
  return c > 1 ? launch_select<kScores, true>(sa, a, t, c, st) : launch_select<kScores, false>(sa, a, t, c, st);
}

cudaError_t kvs_launch_mask_prefix(const SelectArgs& a, const RoundTable& t, cudaStream_t st) {
  const int c = cluster_of(t, a.Hkv, kMaskPairsPerCta, 2 * 148);
  return c > 1 ? launch_select<kMask, true>(StatsTcArgs{}, a, t, c, st) : launch_select<kMask, false>(StatsTcArgs{}, a, t, c, st);
}
