// Attention partials on the tensor cores (tcgen05 + TMEM + TMA), queries on TMEM lanes.
//
// One CTA owns a block of 128 query rows (Q is staged once in shared memory) and a contiguous range
// of 128-slot tiles.  K tiles travel in a three-stage TMA ring and V tiles in one of two stages; per tile one
// thread issues
//   S[q, slot] = Q K_tile^T                         (fp32 in TMEM, three buffers: the logits run two tiles
//                                                    ahead of the P V products, so that a softmax team that
//                                                    has finished a tile finds its next one already formed)
// Two teams of eight softmax warps take alternate tiles, so that one team's arithmetic overlaps
// the other team's waits.  Inside a team the two warps of a TMEM lane quarter own the same 32
// query rows and 64 slot columns each.  A thread reads its logits 16 at a time, forms
// P' = exp(s - m), split into two bf16 terms, and stores them back into the very columns the
// logits came from (16 logits make 8 columns of hi and 8 of lo terms), keeping its part of
// l = sum_j c_j exp(s_j - m): the count bias ln c_j of a merged slot is just the factor c_j in
// that sum.  Another issuing thread then runs
//   O[q, :] += (P'_hi + P'_lo) Vsum_tile            (P' from tensor memory, V as the MN-major operand)
// with the one O accumulating in TMEM across all tiles [Eq. attn_def_vec with merged slots:
// o = sum_j alpha_j Vsum_j / c_j].  At the end the CTA writes (stabiliser, sum, O) as the partial
// of this key range.  Window queries and decode queries use the same kernel.
//
// The stabiliser m of a row is the row's maximum over the CTA's FIRST tile and stays: fp32 sums and
// bf16 terms are floating point, so a later logit that is larger costs no precision until it is
// larger by tens of powers of two.  So no tile but the first needs a maximum, and no warp waits for
// another one.  If a part of l exceeds 2^60 all the same, or the first tile has nothing but logits of -inf
// for a row, the CTA walks its range twice more, once for the true maxima and once with them.  (With a running maximum, exchanged between the two warps of a row and
// between the teams on every tile: 1024 query rows over 131072 slots, 8 heads, 0.83 ms; so: 0.65 ms, 2 000 cycles a
// tile of which the tensor core needs 1 536.)
//
// Eight more warps serve the statistics pass that follows the window attention: tiles are then
// aligned with the round's candidate pairs, and for every pair they form |vbar_l|^2, |vbar_r|^2,
// |vbar_l + vbar_r|^2 and the adjacent-key cosine from the staged rows, so that the statistics
// kernel does not have to touch the rows for it.  The query blocks of a KV head share that work.
#include "kvs_internal.h"
#include "kvs_sm100.cuh"

using namespace sm100;

namespace {

constexpr int kTile = 128;
constexpr int kHalf = 16384;               // [128 rows x 64 bf16], 128-byte swizzle
constexpr int kOperand = 2 * kHalf;
constexpr int kKStages = 3, kVStages = 2;
constexpr int kAhead = 4;                  // tiles requested into L2 ahead of their load
constexpr int kSmemQ = 0, kSmemK = kOperand, kSmemV = kSmemK + kKStages * kOperand;
constexpr int kSmemMisc = kSmemV + kVStages * kOperand;
constexpr int kSoftmaxWarps = 16, kNormWarps = 8;
// Warp 0: TMA, 1: S products, 2-17: softmax, 18-25: pair norms (in calls that form them), the last: P V products.  Decode
// calls are launched without the norm warps: 408 units of three tiles 35.9 -> 34.7 us.
template <bool kNorms> constexpr int kPvWarp = 2 + kSoftmaxWarps + (kNorms ? kNormWarps : 0);
template <bool kNorms> constexpr int kThreads = (kPvWarp<kNorms> + 1) * 32;
constexpr float kSumLimit = 1.152921504606847e18f;   // 2^60: a part of l beyond this asks for another walk
// From here on a logit (log2 units) is scaled and rounded before the stabiliser, which was rounded the same way, is
// subtracted.  One fused multiply-add leaves the product unrounded: two equal logits of 2^24 then differ from
// the stabiliser by up to half a unit, of 1e30 by far more than an exponent holds.
constexpr float kFarLogit = 1048576.f;     // 2^20
constexpr int kSBufs = 3;                  // logit / P' buffers in tensor memory

struct Misc {
  uint64_t kfull[kKStages], vfull[kVStages], kfree[kKStages], vfree[kVStages], sfull[kSBufs], pready[kSBufs][2], pvdone[kSBufs], verdict, qfull, done;
  uint32_t tmem_base;
  int abort_flag, wait_us;                 // (adjacent: the bounded waits read both through one pointer)
  int again;                               // the range is walked again with true maxima
  int k_issued, v_issued;                  // requests of the producer
  alignas(16) float cnt[kSoftmaxWarps][64];   // per warp: the counts of its 64 slots (read as float4)
  float part_max[4][kTile], part_sum[4][kTile];   // the four parts (team x column half) of every row's maximum and sum
};
constexpr int kSmemBytes = kSmemMisc + (int)sizeof(Misc);
static_assert(kSmemBytes <= 232448, "shared memory of one CTA");

constexpr uint32_t kColO = 384;                // TMEM columns: three logit buffers of 128, then O (128)

__device__ __forceinline__ void softmax_barrier() { asm volatile("bar.sync 3, 512;" ::: "memory"); }

// One lane polls, the warp follows.  A failed wait (time-out or abort) only makes the warp skip
// its work: it still goes through the tile loop and the named barriers around it, so that no other
// warp can be left waiting for it.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int lane) {
  int ok = 1;
  if (lane == 0) ok = mbar_wait(bar, parity, abort_flag) ? 1 : 0;
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}
__device__ __forceinline__ void warp_arrive(uint64_t* bar, int lane) {
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void tmem_st_wait() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// |x_l|^2, |x_r|^2 and <x_l, x_r> of the 4 * steps pairs (rows 2 i, 2 i + 1) from row row0 (a multiple of 8) of one
// staged operand, in fp32; lane L gets those of pair pair_of_lane(L), if there is one.  The eight lanes of a
// quarter warp read the eight 16-byte pieces of half a row: with the 128-byte swizzle no bank conflicts.  Plain FMAs,
// two channels per instruction, in a loop that stays rolled.  Small mma.sync products (diagonals of Gram
// matrices) wait for the tensor core behind its own products: 2 400 cycles per operand and tile on four warps,
// where the softmax needs 2 000.  Unrolled FMAs, 1 300, no longer fit the instruction cache together with the
// softmax, and both ran at half their speed (clock64).
__device__ __forceinline__ int pair_of_lane(int lane) { return 4 * ((lane >> 1) & 3) + (lane >> 3); }
__device__ __forceinline__ void pair_dots(const uint8_t* tile, int row0, int steps, int lane, float& ll, float& rr, float& lr) {
  const int c = lane & 7, rl0 = row0 + 2 * (lane >> 3);
  // (the rows of the steps are 8 apart: their swizzle is the same)
  const uint8_t* pl = tile + rl0 * 128 + ((c ^ (rl0 & 7)) << 4);
  const uint8_t* pr = tile + (rl0 + 1) * 128 + ((c ^ ((rl0 + 1) & 7)) << 4);
#pragma unroll 1
  for (int it = 0; it < steps; ++it, pl += 1024, pr += 1024) {
    float2 all = make_float2(0.f, 0.f), arr = all, alr = all;
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      const uint4 l = *reinterpret_cast<const uint4*>(pl + hf * kHalf), r = *reinterpret_cast<const uint4*>(pr + hf * kHalf);
      const uint32_t lw[4] = {l.x, l.y, l.z, l.w}, rw[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 lf = make_float2(bf16lo(lw[i]), bf16hi(lw[i])), rf = make_float2(bf16lo(rw[i]), bf16hi(rw[i]));
        all = __ffma2_rn(lf, lf, all);
        arr = __ffma2_rn(rf, rf, arr);
        alr = __ffma2_rn(lf, rf, alr);
      }
    }
    float o[3] = {all.x + all.y, arr.x + arr.y, alr.x + alr.y};
#pragma unroll
    for (int k = 4; k > 0; k >>= 1)
#pragma unroll
      for (int x = 0; x < 3; ++x) o[x] += __shfl_xor_sync(0xffffffffu, o[x], k);
    if (((lane >> 1) & 3) == it) { ll = o[0]; rr = o[1]; lr = o[2]; }
  }
}
// 1 / sqrt(x) of a sum of squares: the hardware's estimate and a Newton step (the compiler's square root and division took
// 300 cycles a tile).  0 gives a large finite number, and the step is left out where it is not defined (infinity).
__device__ __forceinline__ float rsqrt_newton(float x) {
  const float y = fminf(rsqrtf(x), 1e38f);
  return fmaf(y * 0.5f, fmaxf(fmaf(-x * y, y, 1.f), -1.f), y);
}

template <bool kNorms>
__global__ void __launch_bounds__(kThreads<kNorms>, 1)
flash_partial_tc(const FlashTcArgs a, const RoundTable tab, const __grid_constant__ CUtensorMap tmK,
                 const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmQ) {
  extern __shared__ __align__(1024) uint8_t smem[];
  Misc* misc = reinterpret_cast<Misc*>(smem + kSmemMisc);

  const int seq = blockIdx.z;
  const SeqRound sr = tab.s[seq];
  const int n = sr.n;
  const int h = blockIdx.y;
  const int qblk = blockIdx.x % a.nqblk;
  const int split = blockIdx.x / a.nqblk;
  const int unit = sr.b * a.Hkv + h;
  // (read from one lane, so that the compiler knows the warp index and all that follows from it
  // -- roles, TMEM and barrier addresses -- to be the same in every lane)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  // with pair norms, tile t covers slots [128 t - shift, 128 t - shift + 128): aligned with the pairs
  const int shift = kNorms ? (tab.off & 1) : 0;
  const int ntiles = (n + shift + kTile - 1) / kTile;
  const int t_begin = min(ntiles, split * a.tiles_per_split);
  const int t_end = min(ntiles, t_begin + a.tiles_per_split);
  const int my_tiles = t_end - t_begin;
  kvs_pdl_launch_dependents();
  if (n <= 0) { kvs_pdl_wait(); return; }
  if (smem_u32(smem) & 1023u) {                        // the swizzled tiles need a 1024-byte aligned base
    kvs_pdl_wait();
    if (threadIdx.x == 0 && a.status_dev) atomicExch(a.status_dev, (int)KVS_ERR_CUDA);
    return;
  }
  if (my_tiles <= 0) {
    kvs_pdl_wait();
    // an empty key range still owes its (empty) partial to the combine
    if (warp >= 2 && warp < 6) {
      const int row = (warp & 3) * 32 + lane, m = qblk * 128 + row;
      if (m < a.M) a.part_ml[((size_t)unit * a.splits + split) * a.M + m] = make_float2(-INFINITY, 0.f);
    }
    return;
  }
  // the pair norms of a KV head are shared work of its query blocks: tile t's key cosines belong to block
  // 2 t mod nqblk, its value norms to block 2 t + 1 mod nqblk
  const bool norm_k = kNorms && ((a.nqblk & 1) || !(qblk & 1));
  const bool norm_v = kNorms && ((a.nqblk & 1) || (qblk & 1));
  const int norm_arrivals = norm_k && norm_v ? kNormWarps / 2 : kNormWarps;   // per tile and operand

  if (threadIdx.x == 0) {
    // the K rows of a stage are free once the logits are formed, the V rows only after P V: two
    // rings, so that the next K tiles are requested a whole softmax earlier than the next V tile
    for (int s = 0; s < kKStages; ++s) {
      mbar_init(&misc->kfull[s], 1);
      mbar_init(&misc->kfree[s], norm_k ? 1 + norm_arrivals : 1);   // MMA commit (+ the pair-norm warps)
    }
    for (int s = 0; s < kVStages; ++s) {
      mbar_init(&misc->vfull[s], 1);
      mbar_init(&misc->vfree[s], norm_v ? 1 + norm_arrivals : 1);
    }
    for (int b = 0; b < kSBufs; ++b) {
      mbar_init(&misc->sfull[b], 1);
      mbar_init(&misc->pvdone[b], 1);
      // P' is handed over in two halves (the first and the last 32 slots of every thread's 64), so
      // that the P V products of one half run while the other half is still being written
      for (int hf = 0; hf < 2; ++hf) mbar_init(&misc->pready[b][hf], kSoftmaxWarps / 2);
    }
    mbar_init(&misc->verdict, kSoftmaxWarps);
    mbar_init(&misc->qfull, 1);
    mbar_init(&misc->done, 2);             // all products: the commits of both issuers
    misc->again = 0;
    misc->abort_flag = 0;
    misc->wait_us = (int)a.wait_us;
    mbar_fence_init();
  }
  if (warp == 0 && elect_one()) { prefetch_tmap(&tmK); prefetch_tmap(&tmV); prefetch_tmap(&tmQ); }
  if (warp == 1) tmem_alloc(&misc->tmem_base, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // (everything above runs while the kernel before this one may still be draining)
  kvs_pdl_wait();
  const uint32_t tmem = __shfl_sync(0xffffffffu, misc->tmem_base, 0);   // (uniform for the compiler too)
  volatile int* abort_flag = &misc->abort_flag;
  // test hook: the producer requests no K tile, so that the waits on them run out
  const bool withhold_k = (a.debug_stall & 1u) != 0;
  // Every role walks the range once and then asks whether it is walked twice more (`again`; a range of one tile has
  // its true maxima from the start).  Stages, buffers and phases go by the tile's number over all walks,
  // gi = walk * my_tiles + li.
  auto walks = [&]() -> int {
    if (my_tiles == 1) return 1;
    if (!mbar_wait(&misc->verdict, 0, abort_flag)) return 1;
    return *(volatile int*)&misc->again ? 3 : 1;
  };

  if (warp == 0) {
    // ================================================================ TMA producer
    // one thread streams both rings.  Stages come free in a fixed order (the logits of tile t + 1 are
    // queued before the P V products of tile t), so the thread sleeps on one barrier at a time:
    // K(0), K(1), K(2), V(0), K(3), V(1), ...; every tile is requested into L2 a few tiles ahead
    if (elect_one()) {
      mbar_expect_tx(&misc->qfull, kOperand);
      for (int hf = 0; hf < 2; ++hf)
        tma_load_3d(smem + kSmemQ + hf * kHalf, &tmQ, &misc->qfull, hf * 64, qblk * 128, unit);
      int kgi = 0, vgi = 0, base = 0;                      // (numbers over all walks)
      auto load = [&](const CUtensorMap* tm, uint8_t* dst, uint64_t* full, int li, bool arrives) {
        const int row = (t_begin + li) * kTile - shift;
        if (arrives) {
          mbar_expect_tx(full, kOperand);
          for (int hf = 0; hf < 2; ++hf) tma_load_4d(dst + hf * kHalf, tm, full, hf * 64, row, h, sr.b);
        }
        if (li + kAhead < my_tiles)
          for (int hf = 0; hf < 2; ++hf) tma_prefetch_4d(tm, hf * 64, row + kAhead * kTile, h, sr.b);
      };
      auto load_k = [&]() -> bool {
        const int s = kgi % kKStages;
        if (!mbar_wait(&misc->kfree[s], ((kgi / kKStages) & 1) ^ 1, abort_flag)) return false;
        load(&tmK, smem + kSmemK + s * kOperand, &misc->kfull[s], kgi - base, !withhold_k);
        ++kgi;
        return true;
      };
      auto load_v = [&]() -> bool {
        const int s = vgi % kVStages;
        if (!mbar_wait(&misc->vfree[s], ((vgi / kVStages) & 1) ^ 1, abort_flag)) return false;
        load(&tmV, smem + kSmemV + s * kOperand, &misc->vfull[s], vgi - base, true);
        ++vgi;
        return true;
      };
      bool ok = true;
      for (int walk = 0, n_walks = 1; ok && walk < n_walks; ++walk, base += my_tiles) {
        for (int i = 0; ok && i < min(kKStages - 1, my_tiles); ++i) ok = load_k();
        while (ok && vgi < base + my_tiles) {
          if (kgi < base + my_tiles) ok = load_k();
          if (ok) ok = load_v();
        }
        if (ok && walk == 0) n_walks = walks();
      }
      misc->k_issued = kgi; misc->v_issued = vgi;
    }
  } else if (warp == 1) {
    // ================================================================ issuer of the S products
    // Two threads in two warps feed the tensor pipe, one the logits and one the P V products: a
    // single thread needed 110-125 cycles per product here (it shares its scheduler with four busy
    // softmax warps; its loop was guarded by `lane == 0` then), the pipe 64, and the softmax teams
    // waited for their logits.  Choosing the lane with elect.sync was worth another 3 %.
    if (elect_one()) {
      constexpr uint32_t idesc_s = idesc_bf16(128, 128);                 // Q (K-major) x K tile (K-major)
      const uint64_t qd0 = smem_desc_sw128(smem_u32(smem + kSmemQ), 16, 1024);
      const uint64_t kd0 = smem_desc_sw128(smem_u32(smem + kSmemK), 16, 1024);
      const uint32_t kd_hi = (uint32_t)(kd0 >> 32), qd_lo = (uint32_t)qd0, kd_lo0 = (uint32_t)kd0;
      // The logits of tile gi go to buffer gi mod 3, which last held P' of tile gi - 3: its P V products
      // must be complete (pvdone).  With three buffers the logits run up to three tiles ahead, so that a
      // softmax team that has finished a tile finds the logits of its next one already formed.
      bool ok = mbar_wait(&misc->qfull, 0, abort_flag);
      int end = my_tiles;
      for (int gi = 0; ok && gi < end; ++gi) {
        const int s = gi % kKStages, k = gi / kKStages;    // K stage and its use count
        const int b = gi % kSBufs, u = gi / kSBufs;        // logit buffer and its use count
        if (u > 0 && !mbar_wait(&misc->pvdone[b], (u - 1) & 1, abort_flag)) break;
        if (!mbar_wait(&misc->kfull[s], k & 1, abort_flag)) break;
        tc_fence_after();
        const uint32_t kd_lo = kd_lo0 + s * (kOperand >> 4), ds = tmem + (uint32_t)b * 128;
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t o = ((kk >> 2) * kHalf + (kk & 3) * 32) >> 4;
          if (kk == 0) umma_ss<false>(ds, qd_lo, kd_hi, kd_lo, kd_hi, idesc_s);
          else umma_ss<true>(ds, qd_lo + o, kd_hi, kd_lo + o, kd_hi, idesc_s);
        }
        tc_commit(&misc->sfull[b]);
        tc_commit(&misc->kfree[s]);
        if (gi == my_tiles - 1) end = walks() * my_tiles;
      }
      tc_commit(&misc->done);                              // (behind a walk that broke off, too)
    }
  } else if (warp == kPvWarp<kNorms>) {
    // ================================================================ issuer of the P V products
    if (elect_one()) {
      constexpr uint32_t idesc_o = idesc_bf16(128, 128, false, true);    // P' (K-major) x V tile (MN-major)
      const uint64_t vd0 = smem_desc_sw128(smem_u32(smem + kSmemV), kHalf, 1024);
      const uint32_t vd_hi = (uint32_t)(vd0 >> 32), vd_lo0 = (uint32_t)vd0;
      bool ok = true;
      int end = my_tiles, li = 0;                          // li: the tile's number in this walk
      for (int gi = 0; ok && gi < end; ++gi, li = li + 1 == my_tiles ? 0 : li + 1) {
        const int s = gi % kVStages, ph = (gi / kVStages) & 1;   // V stage and its phase
        const int b = gi % kSBufs, bph = (gi / kSBufs) & 1; // P' buffer and its phase
        if (!mbar_wait(&misc->vfull[s], ph, abort_flag)) ok = false;
        const uint32_t vd_lo = vd_lo0 + s * (kOperand >> 4), ps = tmem + (uint32_t)b * 128;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          if (ok && !mbar_wait(&misc->pready[b][hf], bph, abort_flag)) ok = false;
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int c4 = 0; c4 < 4; ++c4) {
            const int ch = c4 >> 1, k2 = c4 & 1;
            const int kk = 4 * ch + 2 * hf + k2;            // 16-slot step of the tile: slots [16 kk, 16 kk + 16)
#pragma unroll
            for (int hl = 0; hl < 2; ++hl) {
              // A: 16 slots = 8 columns of hi (or, 8 columns further, lo) terms in place of their 16
              // logit columns; B: 16 slots = two 8-row groups of V
              const uint32_t ap = ps + 16 * kk + 8 * hl;
              const uint32_t bl = vd_lo + ((kk * 16 * 128) >> 4);
              if (hf == 0 && c4 == 0 && hl == 0) umma_bf16_ts(tmem + kColO, ap, ((uint64_t)vd_hi << 32) | bl, idesc_o, li > 0 ? 1u : 0u);
              else umma_ts<true>(tmem + kColO, ap, bl, vd_hi, idesc_o);
            }
          }
        }
        if (ok) {
          tc_commit(&misc->vfree[s]);
          tc_commit(&misc->pvdone[b]);
          if (gi == my_tiles - 1) end = walks() * my_tiles;
        }
      }
      tc_commit(&misc->done);
    }
  } else if (warp >= 2 + kSoftmaxWarps) {
    // ================================================================ pair-norm warps
    if (norm_k || norm_v) {
      // A CTA with both operands to do gives the keys to warps 0-3 and the values to warps 4-7, 32 rows of a tile each;
      // one with a single operand gives it to all eight, 16 rows each.  (Every warp sees every tile of its operand:
      // one that skips tiles could take a barrier's phase for an older one.)
      static_assert(kNormWarps == 8, "the split below");
      const int nw = warp - (2 + kSoftmaxWarps);
      const bool both = norm_k && norm_v;
      const int op = both ? nw >> 2 : (norm_v ? 1 : 0);          // 0: keys, 1: values
      const int steps = both ? 4 : 2, row0 = both ? 32 * (nw & 3) : 16 * nw;
      uint64_t* full = op ? misc->vfull : misc->kfull;
      uint64_t* freed = op ? misc->vfree : misc->kfree;
      const int stages = op ? kVStages : kKStages;
      const uint8_t* rows = smem + (op ? kSmemV : kSmemK);
      const int off = tab.off;
      const int32_t* Cn = a.counts + (size_t)unit * a.n_max;
      float* norms = reinterpret_cast<float*>(a.pair_norms + (size_t)unit * a.pair_stride);
      // left slot of this lane's pair; the counts of a slot (no condition: a predicated load is waited for where it is issued)
      int slot_l = t_begin * kTile - shift + row0 + 2 * pair_of_lane(lane);
      const bool has_pair = (lane & 1) == 0 && ((lane >> 1) & 3) < steps;
      auto count_at = [&](int j) { return ldg_here(Cn + min(max(j, 0), n - 1)); };
      int cl_next = count_at(slot_l), cr_next = count_at(slot_l + 1);
      bool ok_all = true;
      int st = 0, ph = 0;
#pragma unroll 1
      for (int li = 0; li < my_tiles; ++li, slot_l += kTile) {
        const int p = (slot_l - off) >> 1;
        const bool mine = (2 * (t_begin + li) + op) % a.nqblk == qblk;
        const int cl = cl_next, cr = cr_next;
        cl_next = count_at(slot_l + kTile); cr_next = count_at(slot_l + kTile + 1);
        if (!warp_wait(full + st, ph, abort_flag, lane)) { ok_all = false; break; }
        float ll = 0.f, rr = 0.f, lr = 0.f;
        if (mine) pair_dots(rows + st * kOperand, row0, steps, lane, ll, rr, lr);
        // the rows are no longer needed here.  (The test is always true: it makes the arrival wait for the loads' results.
        // The barrier of the warp and the arrival order the loads already; this way their data are in registers, too,
        // as in every other place of these kernels where a stage is handed back to the TMA.)
        __syncwarp();
        if (lane == 0 && !(ll < -1.f)) mbar_arrive(freed + st);
        if (++st == stages) { st = 0; ph ^= 1; }
        if (!mine || !has_pair || slot_l < off || p >= sr.P) continue;
        if (op) {
          const float icl = __fdividef(1.f, (float)cl), icr = __fdividef(1.f, (float)cr);   // (small integers)
          const float r2l = ll * icl * icl, r2r = rr * icr * icr;
          norms[4 * (size_t)p] = r2l; norms[4 * (size_t)p + 1] = r2r; norms[4 * (size_t)p + 2] = r2l + r2r + 2.f * lr * icl * icr;
        } else {
          norms[4 * (size_t)p + 3] = lr * fminf(rsqrt_newton(ll) * rsqrt_newton(rr), 1e30f);
        }
      }
      __syncwarp();
      // further walks: the rows are handed back as they come
      if (lane == 0 && ok_all) {
        const int end = walks() * my_tiles;
        for (int gi = my_tiles; gi < end; ++gi) {
          if (!mbar_wait(full + st, ph, abort_flag)) break;
          mbar_arrive(freed + st);
          if (++st == stages) { st = 0; ph ^= 1; }
        }
      }
      __syncwarp();
    }
  } else {
    // ================================================================ softmax warps
    const int team = (warp - 2) >> 3;                     // takes tiles li = team, team + 2, ...
    const int ch = ((warp - 2) >> 2) & 1;                 // 64-slot column half of the tile
    const int row = (warp & 3) * 32 + lane;               // TMEM lane = query row in the block
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const int m = qblk * 128 + row;
    const int last_vis = a.causal ? (n - a.Wq + (m % a.Wq)) : (n - 1);
    const int last_free = min(n - 1, a.causal ? n - a.Wq : n - 1);   // slots up to here need no mask
    const int32_t* Cb = a.counts + (size_t)unit * a.n_max;
    const int part = team * 2 + ch;
    float* cnt = misc->cnt[warp - 2];
    bool alive = true;
    float m_stab = 0.f;                      // the stabiliser (log2 units)
    bool far = false;                        // a row of the warp has one beyond kFarLogit
    // masks the logits of 16 slots from j0 on
    auto mask16 = [&](int j0, float* x) {
      if (j0 >= 0 && j0 + 15 <= last_free) return;
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (j0 + i < 0 || j0 + i > last_vis) x[i] = -INFINITY;
    };
    auto max16 = [&](const float* x) {
      float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
      for (int i = 0; i < 16; ++i) mx[i & 1] = fmaxf(mx[i & 1], x[i]);
      return fmaxf(mx[0], mx[1]);
    };
    // the row's maximum from its four parts (all softmax threads together); false if it has no finite logit
    auto set_stab = [&](float mine) -> bool {
      misc->part_max[part][row] = mine;                    // (read for the last time before the barrier of the verdict)
      softmax_barrier();
      const float mx = fmaxf(fmaxf(misc->part_max[0][row], misc->part_max[1][row]), fmaxf(misc->part_max[2][row], misc->part_max[3][row]));
      m_stab = mx > -INFINITY ? mx * a.scale_log2 : 0.f;
      far = __any_sync(0xffffffffu, fabsf(m_stab) > kFarLogit) != 0;
      return mx > -INFINITY;
    };
    // P' = exp2(scaled logit - m) of 16 slots as hi + lo bf16, two slots per 32-bit column, over the 8 (hi) and
    // 8 (lo) columns in place of the logits.  The hi term is the value cut to bf16 (a byte permute, no
    // conversion); the lo term rounds the exact remainder, so hi + lo carries 16 significant bits.
    // Two slots per instruction: the softmax warps are short of issue slots.
    float2 ls[2];
    auto emit16 = [&](uint32_t col, float* x, const float* cnt16) {
      if (far) {
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] *= a.scale_log2;
      }
      const float sc = far ? 1.f : a.scale_log2;
      const float2 sc2 = make_float2(sc, sc), nm2 = make_float2(-m_stab, -m_stab);
      uint32_t hi[8], lo[8];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float4 ca = *reinterpret_cast<const float4*>(&cnt16[c * 4]);
        const float2 cc[2] = {make_float2(ca.x, ca.y), make_float2(ca.z, ca.w)};
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int i = c * 4 + u * 2;
          const float2 e = __ffma2_rn(make_float2(x[i], x[i + 1]), sc2, nm2);
          const float2 q = make_float2(fast_exp2(e.x), fast_exp2(e.y));
          ls[u] = __ffma2_rn(cc[u], q, ls[u]);
          const uint32_t b0 = __float_as_uint(q.x), b1 = __float_as_uint(q.y);
          hi[c * 2 + u] = __byte_perm(b0, b1, 0x7632);
          const float2 r = __fadd2_rn(q, make_float2(-__uint_as_float(b0 & 0xffff0000u), -__uint_as_float(b1 & 0xffff0000u)));
          lo[c * 2 + u] = pack_bf16(r.x, r.y);
        }
      }
      tmem_st8(col, hi);
      tmem_st8(col + 8, lo);
    };
    // ---- the stabilisers: the rows' maxima over the first tile, 32 columns per thread
    {
      float mx = -INFINITY;
      alive = warp_wait(&misc->sfull[0], 0, abort_flag, lane);
      if (alive) {
        tc_fence_after();
        float xa[16], xb[16];
        tmem_ld16(tmem + lane_addr + part * 32, xa);
        tmem_ld16(tmem + lane_addr + part * 32 + 16, xb);
        tmem_ld_wait();
        const int j0 = t_begin * kTile - shift + part * 32;
        mask16(j0, xa);
        mask16(j0 + 16, xb);
        mx = fmaxf(max16(xa), max16(xb));
        tc_fence_before();
      }
      // A row that sees slots in the first tile, but no logit above -inf, has nothing to go by: its later logits may be
      // of any size, so the range is walked again.  (One that sees none there sees none in this range.)
      if (!set_stab(mx) && alive && max(0, t_begin * kTile - shift) <= last_vis) misc->again = 1;
    }
    int gi_last = 0;
    for (int walk = 0, n_walks = 1; walk < n_walks; ++walk) {
      float mx = -INFINITY;                                // (second walk)
      ls[0] = ls[1] = make_float2(0.f, 0.f);
      // the counts of the warp's slots in its next tile travel meanwhile
      int cn0 = 1, cn1 = 1;
      auto fetch_counts = [&](int li) {
        const int j = (t_begin + li) * kTile - shift + ch * 64 + lane;
        // (outside the sequence P' is 0 and any finite count will do; no condition: a predicated load is waited for
        // where it is issued, which cost 700 cycles a tile)
        cn0 = ldg_here(Cb + min(max(j, 0), n - 1));
        cn1 = ldg_here(Cb + min(max(j + 32, 0), n - 1));
      };
      fetch_counts(team);
      for (int li = team; li < my_tiles; li += 2) {
        const int gi = walk * my_tiles + li;
        const int b = gi % kSBufs, ph = (gi / kSBufs) & 1; // logit buffer and its phase
        const uint32_t scol = tmem + lane_addr + b * 128 + ch * 64;   // this thread's 64 logit columns
        const int tile_row0 = (t_begin + li) * kTile - shift;
        const int j0 = tile_row0 + ch * 64;
        __syncwarp();                                      // (the counts of the tile before have been read)
        cnt[lane] = (float)cn0; cnt[lane + 32] = (float)cn1;
        __syncwarp();
        fetch_counts(li + 2);
        if (alive) alive = warp_wait(&misc->sfull[b], ph, abort_flag, lane);
        if (!alive) continue;
        tc_fence_after();
        if (walk == 1) {
          // the true maxima (what the products make of the logits left in place of P' is never read)
#pragma unroll 1
          for (int c = 0; c < 4; ++c) {
            float x[16];
            tmem_ld16(scol + c * 16, x);
            tmem_ld_wait();
            mask16(j0 + c * 16, x);
            mx = fmaxf(mx, max16(x));
          }
          tc_fence_before();
          warp_arrive(&misc->pready[b][0], lane);
          warp_arrive(&misc->pready[b][1], lane);
          continue;
        }
        // rows of the V tile outside the sequence may hold anything: the team zeroes them
        if (tile_row0 < 0 || tile_row0 + kTile > n) {
          // (the logits run ahead of V by more than its stages: the stage's last use must be over before its barrier's
          // phase says anything about this tile)
          static_assert(kVStages == 2, "the tile that used the stage before");
          if (gi >= 2) alive = warp_wait(&misc->pvdone[(gi - 2) % kSBufs], ((gi - 2) / kSBufs) & 1, abort_flag, lane);
          if (alive) alive = warp_wait(&misc->vfull[gi % kVStages], (gi / kVStages) & 1, abort_flag, lane);
          if (!alive) continue;
          uint8_t* vt = smem + kSmemV + (gi % kVStages) * kOperand;
          for (int it = (threadIdx.x - 64) & 255; it < kTile * 16; it += 256) {
            const int r = it >> 4, c16 = it & 15;
            if (tile_row0 + r < 0 || tile_row0 + r >= n)
              *reinterpret_cast<uint4*>(vt + (c16 >> 3) * kHalf + r * 128 + ((c16 & 7) << 4)) = make_uint4(0, 0, 0, 0);
          }
          fence_proxy_async();                             // the tensor core reads these rows
        }
        // (one copy of the code, run four times: the roles' code has to fit the instruction cache; the other warps cover
        // the latency of the load)
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          float x[16];
          tmem_ld16(scol + c * 16, x);
          tmem_ld_wait();
          mask16(j0 + c * 16, x);
          emit16(scol + c * 16, x, cnt + c * 16);
          if (c & 1) {
            tmem_st_wait();
            tc_fence_before();
            warp_arrive(&misc->pready[b][c >> 1], lane);
          }
        }
      }
      gi_last = (walk + 1) * my_tiles - 1;
      if (walk == 1) set_stab(mx);
      if (walk == 1) continue;
      const float l = (ls[0].x + ls[0].y) + (ls[1].x + ls[1].y);   // this thread's part of l
      misc->part_sum[part][row] = l;                       // (of the first walk, if there are more: not read)
      if (walk == 0 && my_tiles > 1) {
        if (__any_sync(0xffffffffu, !(l < kSumLimit)) && lane == 0) misc->again = 1;
        warp_arrive(&misc->verdict, lane);
      }
      softmax_barrier();
      if (walk == 0 && my_tiles > 1 && *(volatile int*)&misc->again) n_walks = 3;   // (the same for all softmax threads)
    }
    // ---- the stabiliser and sum of this key range: the four parts of a row's sum are added
    if (alive && warp_wait(&misc->pvdone[gi_last % kSBufs], (gi_last / kSBufs) & 1, abort_flag, lane) && part == 0 && m < a.M) {
      const float sum = (misc->part_sum[0][row] + misc->part_sum[1][row]) + (misc->part_sum[2][row] + misc->part_sum[3][row]);
      a.part_ml[((size_t)unit * a.splits + split) * a.M + m] =
          make_float2(sum == 0.f ? -INFINITY : m_stab, sum);   // (a NaN sum is not an empty range)
    }
  }

  // ---- O.  A thread reads 32 channels of its row; written from there, the 16 bytes of 32 rows that a warp stores
  // together lie in 32 lines: 5700 cycles for the 64 KB, a third of the time of a range of two tiles.  They go
  // through the K ring (nobody reads it any more), pieces of 16 bytes exchanged by the row so that neither side has bank
  // conflicts, and out row by row (nine rounds of 8 units from 32 K slots on, events: 304 -> 294 us, six launches of up to 32 tiles 92 ->
  // 86.5, 256 units of 20 tiles 218 -> 212).
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const bool gave_up = *abort_flag != 0;                   // (no wait is left that could set it: the same for all)
  // Nothing may be in flight when the CTA leaves: its shared and tensor memory are the next CTA's from then on.  Whole walks
  // have waited for their copies and products, but for the last arrivals that hand the stages back; behind one that
  // broke off, in whichever role and after whichever request, any copy and any product may be under way.
  if (threadIdx.x == 0) {
    const int nk = misc->k_issued, nv = misc->v_issued;
    mbar_drain(&misc->done, 0);
    if (gave_up) mbar_drain(&misc->qfull, 0);
    if (!(gave_up && withhold_k))
      for (int gi = max(0, nk - kKStages); gi < nk; ++gi)
        mbar_drain(gave_up ? &misc->kfull[gi % kKStages] : &misc->kfree[gi % kKStages], (gi / kKStages) & 1);
    for (int gi = max(0, nv - kVStages); gi < nv; ++gi)
      mbar_drain(gave_up ? &misc->vfull[gi % kVStages] : &misc->vfree[gi % kVStages], (gi / kVStages) & 1);
  }
  if (warp >= 2 && warp < 2 + kSoftmaxWarps && !gave_up) {
    const int part = (warp - 2) >> 2, row = (warp & 3) * 32 + lane;
    uint8_t* stage = smem + kSmemK;
    float ov[32];
    tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + kColO + part * 32, ov);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 8; ++i)
      *reinterpret_cast<float4*>(stage + row * (KVS_D * 4) + (((part * 8 + i) ^ (row & 7)) << 4)) =
          make_float4(ov[4 * i], ov[4 * i + 1], ov[4 * i + 2], ov[4 * i + 3]);
    softmax_barrier();
    const int rows = min(kTile, a.M - qblk * kTile);
    float4* po = reinterpret_cast<float4*>(a.part_o + (((size_t)unit * a.splits + split) * a.M + qblk * kTile) * KVS_D);
#pragma unroll
    for (int r = warp - 2; r < kTile; r += kSoftmaxWarps)
      if (r < rows) po[r * (KVS_D / 4) + lane] = *reinterpret_cast<const float4*>(stage + r * (KVS_D * 4) + ((lane ^ (r & 7)) << 4));
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (threadIdx.x == 0 && gave_up && a.status_dev) atomicExch(a.status_dev, (int)KVS_ERR_TIMEOUT);
}

}  // namespace

cudaError_t kvs_launch_flash_tc(const FlashTcArgs& a, const RoundTable& t, const CUtensorMap& tmK,
                                const CUtensorMap& tmV, const CUtensorMap& tmQ, cudaStream_t st) {
  static KvsPerDeviceOnce configured;
  cudaError_t ce = configured.run([] {
    for (auto k : {flash_partial_tc<false>, flash_partial_tc<true>}) {
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  });
  if (ce != cudaSuccess) return ce;
  dim3 grid(a.nqblk * a.splits, a.Hkv, t.nseq);
  const bool norms = a.pair_norms != nullptr;
  return kvs_launch_chained(norms ? flash_partial_tc<true> : flash_partial_tc<false>, grid,
                            dim3(norms ? kThreads<true> : kThreads<false>), kSmemBytes, st, a, t, tmK, tmV, tmQ);
}
