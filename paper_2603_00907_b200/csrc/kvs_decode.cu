// Attention of a few new query rows over a merged cache (the decode step of a generation): at most
// 16 rows per KV head, i.e. group * n_new <= 16 [Eq. attn_def_vec with merged slots].
//
// Bound by HBM: every K and Vsum row is used for one handful of multiply-adds, so what counts is bytes
// in flight and short set-up.  (A 128-row tcgen05 tile is 1 to 12 % full here, and its fixed costs --
// TMEM, 736 threads, a combine kernel -- took 14 us where the 8 MB of one sequence need one.)
// Each warp walks blocks of 16 slots on its own: its ring of three blocks in shared memory is filled by
// TMA (no barrier between warps; two CTAs of four warps keep 192 KB of an SM in flight) and read as
// mma.sync m16n8k16 fragments, slots resp. channels on the 16 rows and queries on the 8 columns:
//   S^T[slot, q] = K Q^T      the channel order of a contraction is free: a lane's 16-byte piece of a
//                             K row and of a Q row hold the same channels, two products' worth
//   P' = exp2(S - m)          per warp; m moves only when it is outgrown by more than 2^8
//   O^T[chan, q] += V^T P'^T  two V rows are zipped with byte permutes, P'^T comes from movmatrix, and P'
//                             enters as hi + lo bf16 terms (16 significant bits)
// The warps of a cluster of CTAs share a (sequence, KV head) unit block by block; they merge their
// (m, l, O) through shared and distributed shared memory and write the output, with no second
// kernel.  A unit that needs more than one cluster leaves a partial per cluster for combine_partials.
// Measured (8 KV heads, group 4, one new token), before -> after: one sequence of 2048 slots 13.3 -> 7.4 us
// on the GPU; 32 sequences of 512-8192 slots (610 MB) 162 -> 93 us, 6.5 TB/s; 16 sequences of 8192 slots with
// 16 rows 135 -> 90 us.  Loads straight into registers reached 4.9-5.5 TB/s, lane-private cp.async 4.9.
#include <cooperative_groups.h>

#include <mutex>

#include "kvs_internal.h"
#include "kvs_sm100.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kWarps = 4;                  // per CTA
constexpr int kBlock = 16;                 // slots per step of a warp
constexpr int kStages = 3;                 // blocks of a warp in flight
constexpr int kSub = kBlock * 128;         // [16 rows x 64 bf16], 128-byte swizzle
constexpr int kStageBytes = 4 * kSub;      // channels 0-63 and 64-127 of K, then of Vsum
constexpr int kWarpBytes = kStages * kStageBytes;
constexpr int kSmemBytes = kWarps * kWarpBytes;
constexpr float kRescaleGap = 8.f;         // log2 units
// The stabiliser before any logit.  Finite, so that a block whose logits are all -inf gives weights of 0 (-inf - (-inf)
// would be NaN), and the lowest value, so that every finite logit moves it.  What has it still at the end is
// merged like the rest: nothing or zeros are added, and a NaN stays.
constexpr float kNoMax = -3.402823466e38f;
// The stabiliser is put a little above the maximum.  At the maximum P' would be exactly 1, its lo term 0, and 0 times an
// infinite value NaN: one row in sixteen that sees an infinite value had its block's maximum there.
constexpr float kAbove = 0.01f;

__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1) {
  // (volatile: a stage's next request stays behind the products of its rows)
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t transpose8(uint32_t v) {     // 8 x 8 matrix of 16-bit words over the warp
  uint32_t r;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
  return r;
}
// A count travels with its block (a load into a register would be waited for one block later at the latest).
__device__ __forceinline__ void copy4(void* dst, const int32_t* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sm100::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory"); }

// Lane 4 g + t reads, of a block of 16 slots: K rows g and g + 8, 16-byte chunks 2 t, 2 t + 1 of either
// half; V rows 2 t, 2 t + 1, 2 t + 8, 2 t + 9, chunk g of either half.  With the 128-byte swizzle the eight
// lanes of a quarter warp then touch eight different 16-byte columns: no bank conflicts.
__device__ __forceinline__ uint4 chunk_of(const uint8_t* sub, int row, int chunk) {
  return *reinterpret_cast<const uint4*>(sub + row * 128 + ((chunk ^ (row & 7)) << 4));
}

// kTiles tiles of 8 query columns.  kFour: at most four rows, which take the columns 0-3 and again 4-7:
// the second product then forms the hi terms' part of O in the one half and the lo terms' in the other.
template <int kTiles, bool kFour>
__global__ void __launch_bounds__(kWarps * 32, 2)
decode_rows_kernel(const DecodeArgs a, const RoundTable tab, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmV) {
  constexpr int kRows = 8 * kTiles;
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ uint64_t s_full[kWarps][kStages];
  __shared__ int32_t s_cnt[kWarps][kStages][kBlock];
  __shared__ int s_ctl[2];                               // abort flag, time limit of a wait (microseconds)
  __shared__ float s_m[kWarps][kRows], s_l[kWarps][kRows];
  __shared__ float s_cm[kRows], s_cl[kRows];             // of the CTA: maximum and sum
  kvs_pdl_launch_dependents();
  if (sm100::smem_u32(smem) & 1023u) {                    // the swizzled tiles need a 1024-byte aligned base (the same in every CTA)
    kvs_pdl_wait();
    if (threadIdx.x == 0 && a.status_dev) atomicExch(a.status_dev, (int)KVS_ERR_CUDA);
    return;
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < kWarps * kStages; ++i) sm100::mbar_init(&s_full[0][i], 1);
    s_ctl[0] = 0;
    s_ctl[1] = (int)a.wait_us;
    sm100::mbar_fence_init();
  }
  __syncthreads();
  kvs_pdl_wait();
  cg::cluster_group cluster = cg::this_cluster();
  const int ctas = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int split = blockIdx.x / ctas;
  const SeqRound sr = tab.s[blockIdx.z];
  const int n = sr.n;
  const int unit = sr.b * a.Hkv + blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int32_t* Cb = a.counts + (size_t)unit * a.n_max;

  // blocks of this cluster, dealt out to its warps in turn
  const int nblocks = (n + kBlock - 1) / kBlock;
  const int per_split = (nblocks + a.splits - 1) / a.splits;
  const int b_end = min(nblocks, (split + 1) * per_split);
  const int b_step = ctas * kWarps;
  int b = split * per_split + rank * kWarps + warp;

  uint8_t* mine = smem + warp * kWarpBytes;              // this warp's ring
  uint64_t* full = s_full[warp];
  volatile int* ctl = s_ctl;
  const bool withhold = (a.debug_stall & 1u) != 0;        // test hook: nothing is requested, so that the waits run out
  auto request = [&](int blk, int stage) {
    if (blk < b_end) {
      if (lane < kBlock) copy4(&s_cnt[warp][stage][lane], Cb + min(blk * kBlock + lane, n - 1));
      if (lane == 0 && !withhold) {
        uint8_t* dst = mine + stage * kStageBytes;
        sm100::mbar_expect_tx(&full[stage], kStageBytes);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          sm100::tma_load_4d(dst + hf * kSub, &tmK, &full[stage], hf * 64, blk * kBlock, blockIdx.y, sr.b);
          sm100::tma_load_4d(dst + (2 + hf) * kSub, &tmV, &full[stage], hf * 64, blk * kBlock, blockIdx.y, sr.b);
        }
      }
    }
    copy_commit();                                       // (empty groups at the end keep the count right)
  };
  if (lane == 0) { sm100::prefetch_tmap(&tmK); sm100::prefetch_tmap(&tmV); }
  for (int s = 0; s < kStages; ++s) request(b + s * b_step, s);
  // query rows as B fragments: lane 4 g + t holds row g of each tile
  uint32_t q[kTiles][4][4];
#pragma unroll
  for (int nt = 0; nt < kTiles; ++nt) {
    const int m = kFour ? g & 3 : nt * 8 + g;
    const uint4* p = reinterpret_cast<const uint4*>(a.q + ((size_t)unit * a.M + min(m, a.M - 1)) * KVS_D) + 2 * t;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint4 v = m < a.M ? p[(i >> 1) * 8 + (i & 1)] : make_uint4(0, 0, 0, 0);
      q[nt][i][0] = v.x; q[nt][i][1] = v.y; q[nt][i][2] = v.z; q[nt][i][3] = v.w;
    }
  }
  // O^T: tile jb holds channels 8 g + jb (elements 0, 1) and 64 + 8 g + jb (2, 3) of queries 2 t and 2 t + 1
  float o[kTiles][8][4], l[kTiles][2], m_run[kTiles][2];
#pragma unroll
  for (int nt = 0; nt < kTiles; ++nt) {
#pragma unroll
    for (int jb = 0; jb < 8; ++jb)
#pragma unroll
      for (int i = 0; i < 4; ++i) o[nt][jb][i] = 0.f;
    l[nt][0] = l[nt][1] = 0.f;
    m_run[nt][0] = m_run[nt][1] = kNoMax;
  }

  int stage = 0;
  uint32_t phase = 0;
  for (; b < b_end; b += b_step) {
    int good = 1;
    if (lane == 0) good = sm100::mbar_wait(&full[stage], phase, ctl) ? 1 : 0;
    copy_wait<kStages - 1>();
    if (!__shfl_sync(0xffffffffu, good, 0)) break;
    __syncwarp();                                        // the other lanes' counts are visible
    const uint8_t* st = mine + stage * kStageBytes;
    const int j0 = b * kBlock;
    const bool ok0 = j0 + g < n, ok1 = j0 + g + 8 < n;
    const float c0 = (float)s_cnt[warp][stage][g], c1 = (float)s_cnt[warp][stage][g + 8];
    float s[kTiles][4];
    {
      uint4 k0[4], k1[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        k0[i] = chunk_of(st + (i >> 1) * kSub, g, 2 * t + (i & 1));
        k1[i] = chunk_of(st + (i >> 1) * kSub, g + 8, 2 * t + (i & 1));
      }
#pragma unroll
      for (int nt = 0; nt < kTiles; ++nt) {
        float e[4] = {0.f, 0.f, 0.f, 0.f};               // two chains of products
#pragma unroll
        for (int i = 0; i < 4; ++i) s[nt][i] = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          mma_16816(s[nt], k0[i].x, k1[i].x, k0[i].y, k1[i].y, q[nt][i][0], q[nt][i][1]);
          mma_16816(e, k0[i].z, k1[i].z, k0[i].w, k1[i].w, q[nt][i][2], q[nt][i][3]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) s[nt][i] += e[i];
      }
    }
    uint32_t bh[kTiles][2], bl[kTiles][2];               // P'^T as B fragments
#pragma unroll
    for (int nt = 0; nt < kTiles; ++nt) {
#pragma unroll
      for (int i = 0; i < 4; ++i) s[nt][i] = (i < 2 ? ok0 : ok1) ? s[nt][i] * a.scale_log2 : -INFINITY;
      // the stabilisers of the two query columns
      const float mx0 = fmaxf(s[nt][0], s[nt][2]), mx1 = fmaxf(s[nt][1], s[nt][3]);
      if (__any_sync(0xffffffffu, mx0 > m_run[nt][0] + kRescaleGap || mx1 > m_run[nt][1] + kRescaleGap)) {
        float mn[2] = {mx0, mx1};
#pragma unroll
        for (int k = 4; k < 32; k <<= 1) {
          mn[0] = fmaxf(mn[0], __shfl_xor_sync(0xffffffffu, mn[0], k));
          mn[1] = fmaxf(mn[1], __shfl_xor_sync(0xffffffffu, mn[1], k));
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const float m_new = fmaxf(mn[u] + kAbove, m_run[nt][u]);
          const float f = fast_exp2(m_run[nt][u] - m_new);
          l[nt][u] *= f;
#pragma unroll
          for (int jb = 0; jb < 8; ++jb) { o[nt][jb][u] *= f; o[nt][jb][2 + u] *= f; }
          m_run[nt][u] = m_new;
        }
      }
      float p[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) p[i] = fast_exp2(s[nt][i] - m_run[nt][i & 1]);
      l[nt][0] = fmaf(c0, p[0], fmaf(c1, p[2], l[nt][0]));
      l[nt][1] = fmaf(c0, p[1], fmaf(c1, p[3], l[nt][1]));
      // hi: the value cut to bf16; lo: the rounded remainder.  [slot, q] -> [q, slot] for the second product
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint32_t w0 = __float_as_uint(p[2 * u]), w1 = __float_as_uint(p[2 * u + 1]);
        const __nv_bfloat162 lo = __floats2bfloat162_rn(p[2 * u] - __uint_as_float(w0 & 0xffff0000u),
                                                        p[2 * u + 1] - __uint_as_float(w1 & 0xffff0000u));
        const uint32_t hi_w = __byte_perm(w0, w1, 0x7632), lo_w = *reinterpret_cast<const uint32_t*>(&lo);
        bh[nt][u] = transpose8(kFour && t >= 2 ? lo_w : hi_w);
        if (!kFour) bl[nt][u] = transpose8(lo_w);
      }
    }
    uint4 vr[4][2];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int row = 2 * t + (r & 1) + 8 * (r >> 1);
      vr[r][0] = chunk_of(st + 2 * kSub, row, g);
      vr[r][1] = chunk_of(st + 3 * kSub, row, g);
      if (j0 + kBlock > n && j0 + row >= n) vr[r][0] = vr[r][1] = make_uint4(0, 0, 0, 0);   // (may hold anything)
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      uint32_t v[4][2];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf)
          v[r][hf] = w == 0 ? vr[r][hf].x : w == 1 ? vr[r][hf].y : w == 2 ? vr[r][hf].z : vr[r][hf].w;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const uint32_t sel = e ? 0x7632 : 0x5410;
        const uint32_t a0 = __byte_perm(v[0][0], v[1][0], sel), a1 = __byte_perm(v[0][1], v[1][1], sel);
        const uint32_t a2 = __byte_perm(v[2][0], v[3][0], sel), a3 = __byte_perm(v[2][1], v[3][1], sel);
#pragma unroll
        for (int nt = 0; nt < kTiles; ++nt) {
          mma_16816(o[nt][2 * w + e], a0, a1, a2, a3, bh[nt][0], bh[nt][1]);
          if (!kFour) mma_16816(o[nt][2 * w + e], a0, a1, a2, a3, bl[nt][0], bl[nt][1]);
        }
      }
    }
    // The block after the next ones takes the stage.  The request stands behind the products that use the stage's rows:
    // a barrier of the warp orders the loads' issue, the products wait for their data.  (In front of the products: 8
    // units of 8192 slots 13.7 against 13.9 us, 256 units 158.8 against 158.6.)
    __syncwarp();
    request(b + kStages * b_step, stage);
    if (++stage == kStages) { stage = 0; phase ^= 1; }
  }
  if (ctl[0] && lane == 0 && !withhold) {
    // a wait ran out: give the copies in flight a bounded time to land before the CTA leaves
    for (int s = 0; s < kStages && b + s * b_step < b_end; ++s) {
      const int st = (stage + s) % kStages;
      sm100::mbar_drain(&full[st], phase ^ (stage + s >= kStages ? 1u : 0u));
    }
  }
  copy_wait<0>();
  float* o_mine = reinterpret_cast<float*>(mine);        // [kRows][128]: the ring is empty

  // ---- the warps of the CTA: common maximum, sums of l and O
#pragma unroll
  for (int nt = 0; nt < kTiles; ++nt)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
#pragma unroll
      for (int k = 4; k < 32; k <<= 1) l[nt][u] += __shfl_xor_sync(0xffffffffu, l[nt][u], k);
      if (g == 0) { s_m[warp][nt * 8 + 2 * t + u] = m_run[nt][u]; s_l[warp][nt * 8 + 2 * t + u] = l[nt][u]; }
    }
  __syncthreads();
  if (threadIdx.x < kRows) {
    float mx = -INFINITY, sum = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) mx = fmaxf(mx, s_m[w][threadIdx.x]);
#pragma unroll
    for (int w = 0; w < kWarps; ++w) sum = fmaf(s_l[w][threadIdx.x], fast_exp2(s_m[w][threadIdx.x] - mx), sum);
    s_cm[threadIdx.x] = mx; s_cl[threadIdx.x] = sum;
  }
  __syncthreads();
  if (kFour) {
#pragma unroll
    for (int jb = 0; jb < 8; ++jb)
#pragma unroll
      for (int i = 0; i < 4; ++i) o[0][jb][i] += __shfl_xor_sync(0xffffffffu, o[0][jb][i], 2);
  }
#pragma unroll
  for (int nt = 0; nt < kTiles; ++nt)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (kFour && t >= 2) continue;
      const int row = nt * 8 + 2 * t + u;
      const float f = fast_exp2(m_run[nt][u] - s_cm[row]);
#pragma unroll
      for (int hf = 0; hf < 2; ++hf)
#pragma unroll
        for (int x = 0; x < 2; ++x)
          *reinterpret_cast<float4*>(o_mine + row * KVS_D + 64 * hf + 8 * g + 4 * x) =
              make_float4(o[nt][4 * x][2 * hf + u] * f, o[nt][4 * x + 1][2 * hf + u] * f,
                          o[nt][4 * x + 2][2 * hf + u] * f, o[nt][4 * x + 3][2 * hf + u] * f);
    }
  __syncthreads();
  for (int i = threadIdx.x; i < a.M * (KVS_D / 4); i += kWarps * 32) {
    float4* d = reinterpret_cast<float4*>(smem) + i;
    float4 acc = *d;
#pragma unroll
    for (int w = 1; w < kWarps; ++w) {
      const float4 v = reinterpret_cast<const float4*>(smem + w * kWarpBytes)[i];
      acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
    *d = acc;
  }
  // ---- the CTAs of the cluster: each one merges its share of the rows' channels
  cluster.sync();
  const int quads = a.M * (KVS_D / 4);                     // float4 columns of all rows
  for (int i = rank * (kWarps * 32) + threadIdx.x; i < quads; i += ctas * kWarps * 32) {
    const int row = i >> 5, c4 = i & 31;
    float mx = -INFINITY;
    for (int r = 0; r < ctas; ++r) mx = fmaxf(mx, *cluster.map_shared_rank(&s_cm[row], r));
    float sum = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int r = 0; r < ctas; ++r) {
      const float f = fast_exp2(*cluster.map_shared_rank(&s_cm[row], r) - mx);
      const float4 v = *cluster.map_shared_rank(reinterpret_cast<float4*>(smem) + i, r);
      sum = fmaf(*cluster.map_shared_rank(&s_cl[row], r), f, sum);
      acc.x = fmaf(v.x, f, acc.x); acc.y = fmaf(v.y, f, acc.y);
      acc.z = fmaf(v.z, f, acc.z); acc.w = fmaf(v.w, f, acc.w);
    }
    if (a.splits > 1) {
      const size_t pidx = ((size_t)unit * a.splits + split) * a.M + row;
      *reinterpret_cast<float4*>(a.part_o + pidx * KVS_D + 4 * c4) = acc;
      if (c4 == 0) a.part_ml[pidx] = make_float2(mx, sum);
    } else {
      const float inv = 1.f / sum;
      const __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x * inv, acc.y * inv), hi = __floats2bfloat162_rn(acc.z * inv, acc.w * inv);
      const size_t orow = (size_t)unit * a.M + row;
      *reinterpret_cast<uint2*>(a.out + orow * KVS_D + 4 * c4) =
          make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
      if (c4 == 0 && a.lse) a.lse[orow] = (mx + log2f(sum)) * 0.6931471805599453f;
    }
  }
  cluster.sync();                                          // no CTA leaves while its shared memory is read
  if (threadIdx.x == 0 && ctl[0] && a.status_dev) atomicExch(a.status_dev, (int)KVS_ERR_TIMEOUT);
}

template <int kTiles, bool kFour>
cudaError_t configure_rows() {
  static KvsPerDeviceOnce configured;
  return configured.run([] {
    return cudaFuncSetAttribute(decode_rows_kernel<kTiles, kFour>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  });
}

template <int kTiles, bool kFour>
cudaError_t launch_rows(const DecodeArgs& a, const RoundTable& t, const CUtensorMap& tmK, const CUtensorMap& tmV, int ctas,
                        cudaStream_t st) {
  cudaError_t e = configure_rows<kTiles, kFour>();
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(ctas * a.splits), (unsigned)a.Hkv, (unsigned)t.nseq);
  cfg.blockDim = dim3(kWarps * 32);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)ctas;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, decode_rows_kernel<kTiles, kFour>, a, t, tmK, tmV);
}

}  // namespace

// Clusters of 1 to 8 CTAs that are resident at once (entry k: of k CTAs): two CTAs fit an SM, but a cluster has to find its
// place in one group of SMs, and the groups are not all of one size (one B200: 296, 148, 93, 71, 56, 45, 37 and 33
// clusters).  Asked once per device for the kernel of the most rows; all of them are bound by shared memory.
const int* kvs_decode_resident_clusters() {
  struct Table { std::atomic<int> known; int n[KVS_DECODE_CLUSTER + 1]; };
  static Table tables[64] = {};
  static std::mutex mutex;
  static const int unknown[KVS_DECODE_CLUSTER + 1] = {0, 256, 128, 85, 64, 51, 42, 36, 32};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return unknown;
  Table& t = tables[dev];
  if (t.known.load(std::memory_order_acquire)) return t.n;
  std::lock_guard<std::mutex> lock(mutex);
  for (int k = 1; k <= KVS_DECODE_CLUSTER; ++k) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)k);
    cfg.blockDim = dim3(kWarps * 32);
    cfg.dynamicSmemBytes = kSmemBytes;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)k;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (configure_rows<2, false>() != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, decode_rows_kernel<2, false>, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();                                  // (the launch itself reports what is wrong)
      return unknown;
    }
    t.n[k] = n;
  }
  t.known.store(1, std::memory_order_release);
  return t.n;
}

cudaError_t kvs_launch_decode_rows(const DecodeArgs& a, const RoundTable& t, const CUtensorMap& tmK,
                                   const CUtensorMap& tmV, int ctas, cudaStream_t st) {
  if (a.M <= 4) return launch_rows<1, true>(a, t, tmK, tmV, ctas, st);
  return a.M <= 8 ? launch_rows<1, false>(a, t, tmK, tmV, ctas, st) : launch_rows<2, false>(a, t, tmK, tmV, ctas, st);
}
