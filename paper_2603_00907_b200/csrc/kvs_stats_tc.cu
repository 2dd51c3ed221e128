// Hessian statistics on the tensor cores (tcgen05 + TMEM + TMA), candidate pairs on TMEM lanes.
//
// One CTA owns a block of 128 window queries (Q, and the attention output O split into two
// bf16 terms, stay in shared memory) and walks a range of tiles of 128 candidate pairs.
// A 5-D view of the cache, [128, parity, slot/2, head, sequence], lets TMA bring the left
// members and the right members of the 128 pairs as two separate row tiles, so that TMEM
// lane p holds everything of pair p.  For each step of up to 64 queries
//   S_l = K_l Q^T, S_r = K_r Q^T                    (logits, fp32 in TMEM)
//   T_l = Vsum_l (O_hi + O_lo)^T, T_r likewise      (value/output inner products)
// go into one of two TMEM buffers; while the statistics warps reduce one step, the tensor
// core fills the other buffer with the next (of the same tile, or of the next tile where a block has
// no more than 64 queries: 16 x 8 units of 16 K pairs and 64 window rows 233 -> 198 us).  Two threads (in two warps, each chosen with elect.sync) issue the
// products, one the chains of the left members and one those of the right members: one thread
// alone measured 2 % slower.  Each statistics thread owns one pair
// and a share of the queries and reduces, in registers and with no cross-lane traffic,
//   A_j   = sum_q alpha_qj
//   N1_j  = sum_q alpha |1 - 2 alpha| |vbar_j - o_q|                    [Eqs. c11_def, c22_def]
//   N12_p = sum_q alpha_j alpha_j+1 |vbar_j + vbar_j+1 - 2 o_q|         [Eq. c12_def]
// with |vbar_j - o_q|^2 = |vbar_j|^2 - 2 T_jq / c_j + |o_q|^2.  The probability matrix never
// leaves the SM.  The row norms |vbar|^2, |vbar_l + vbar_r|^2 and the adjacent-key cosine of
// every pair come from the attention pass that precedes this kernel (it streams the same rows).
// Every (query block, statistics group) writes its five sums per pair as a partial; the
// selection (kvs_select.cu) adds the partials in a fixed order and forms score and the merge weight of
// Eq. kstar_final (deterministic, no atomics, no hand-over between warps inside the tile loop).
// A second instantiation serves the exact weight modes: a supplied loss gradient E (one row per
// window query) takes the place of the attention output in the T products, and the statistics
// warps sum the signed scalars g_ij = E^T c_ij instead of the norms [Section 4.2, text before
// Eq. h_rank1_unified; Eq. kstar_weight_final_rewrite].
// What bounds it (256 units of 16 K pairs, 128 queries each, 906 us, 6500 cycles a tile): the special-function
// pipe needs 5120 cycles a tile (the arithmetic alone, without waits, runs in 5500), the operand reads of
// the products 4600 of the shared-memory pipe's cycles, and the chip holds 1.6 to 1.7 GHz under this mix.  Tried
// and slower: operands of the pairs copied to tensor memory (products half as long, 32 queries a step,
// sixteen statistics warps: +4 %), a team of warps for each buffer (+3 % with sixteen, +8 % with eight), one of the
// two exponentials by a polynomial on the FMA pipe (+1 to 4 %).
// Every synchronisation is an mbarrier with a bounded wait, so a warp that gives up can never
// leave another one stuck.
#include "kvs_internal.h"
#include "kvs_sm100.cuh"

using namespace sm100;

namespace {

constexpr int kPairs = 128;                // candidate pairs per tile = TMEM lanes
constexpr int kQB = 128;                   // queries per CTA
constexpr int kQH = 64;                    // queries per accumulator buffer, at most
constexpr int kHalf = 16384;               // bytes of a [128 rows x 64 bf16] swizzled sub-tile
constexpr int kOperand = 2 * kHalf;        // a [128 x 128] bf16 operand
constexpr int kSmemQ = 0, kSmemOhi = kOperand, kSmemOlo = 2 * kOperand;
constexpr int kSmemKl = 3 * kOperand, kSmemKr = 4 * kOperand, kSmemVl = 5 * kOperand, kSmemVr = 6 * kOperand;
constexpr int kSmemMisc = 7 * kOperand;
constexpr int kGroups = KVS_STATS_GROUPS;  // statistics groups: a group reduces a share of the queries of every step
constexpr int kChunk = 8;                  // queries per round of TMEM loads
constexpr int kStatWarps = 4 * kGroups;
constexpr int kIssuers = 2;
constexpr int kFirstStat = 1 + kIssuers;   // warp 0: TMA, warps 1-2: product issuers, then the statistics warps
constexpr int kThreads = (kFirstStat + kStatWarps) * 32;
// bounds the registers to 96: the CTAs of the finalize kernel (256 threads of 40 registers) then fit beside a
// statistics CTA and are launched while it runs
constexpr int kBoundThreads = 544;
static_assert(KVS_STATS_GROUPS == kGroups, "the launcher sizes the partials with KVS_STATS_GROUPS");

struct Misc {
  uint64_t kfull, vfull, kfree, vfree, tfull[2], tfree[2], qfull, qfree, cfull, cfree, done;
  uint32_t tmem_base;
  int abort_flag, wait_us;                 // (adjacent: the bounded waits read both through one pointer)
  uint32_t k_issued, v_issued, q_issued, c_issued;   // requests of the producer
  // per two queries (2k, 2k+1) of the block: (c_2k, c_2k+1, h_2k, h_2k+1) with c = -(max + log2 Z) and
  // h = |o|^2 (or <E, o>): neighbours sit side by side for the packed two-float arithmetic
  alignas(16) float qconst[2 * kQB];
};
constexpr int kSmemBytes = kSmemMisc + (int)sizeof(Misc);
static_assert(kSmemBytes <= 232448, "shared memory of one CTA");

// One lane waits, the warp follows.  (Polling in a tight loop instead of letting the hardware
// suspend the lane measured the same: the statistics warps' waits, about 250 cycles per half, are
// real waits for the tensor core, not wake-up latency.)
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int lane) {
  int ok = 1;
  if (lane == 0) ok = mbar_wait(bar, parity, abort_flag) ? 1 : 0;
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}
__device__ __forceinline__ void warp_arrive(uint64_t* bar, int lane) {
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}

__device__ __forceinline__ float fast_sqrt(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// The segments a group of CTAs walks: tiles of one (sequence, KV head) unit after another.
struct Walk {
  int left, seq, h, t, count;              // tiles not yet handed out; the segment: unit, first tile, tiles
  int seq_next, h_next, t_next;
  static __device__ __forceinline__ int tiles_of(const RoundTable& tab, int seq) {
    return tab.s[seq].n > 0 ? (tab.s[seq].P + kPairs - 1) / kPairs : 0;
  }
  // a range of `tiles` of the unit (blockIdx.z, blockIdx.y)
  static __device__ __forceinline__ Walk range(const RoundTable& tab, int split, int tiles) {
    Walk w;
    w.seq_next = blockIdx.z;
    w.h_next = blockIdx.y;
    w.t_next = split * tiles;
    w.left = min(tiles, tiles_of(tab, w.seq_next) - w.t_next);
    return w;
  }
  // an equal share of the tiles of all units; the first `extra` groups take one more
  static __device__ __forceinline__ Walk share(const RoundTable& tab, int Hkv, int group, int tiles, int extra) {
    Walk w;
    int first = group * tiles + min(group, extra);
    w.left = tiles + (group < extra ? 1 : 0);
    int nt = tiles_of(tab, 0);
    for (w.seq_next = 0; first >= nt * Hkv && w.seq_next + 1 < tab.nseq; nt = tiles_of(tab, ++w.seq_next)) first -= nt * Hkv;
    w.h_next = nt > 0 ? first / nt : 0;
    w.t_next = first - w.h_next * nt;
    return w;
  }
  // (divisions leave the unit in per-lane registers: read from one lane, the compiler keeps it and all that
  // follows from it in uniform ones; for whole warps only)
  __device__ __forceinline__ void make_uniform() {
    seq = __shfl_sync(0xffffffffu, seq, 0);
    h = __shfl_sync(0xffffffffu, h, 0);
    t = __shfl_sync(0xffffffffu, t, 0);
    count = __shfl_sync(0xffffffffu, count, 0);
  }
  __device__ __forceinline__ bool next(const RoundTable& tab, int Hkv) {
    if (left <= 0) return false;
    while (h_next == Hkv || tiles_of(tab, seq_next) == 0) {   // (tiles are left, so a unit that has some follows)
      ++seq_next;
      h_next = 0;
    }
    const int nt = tiles_of(tab, seq_next);
    seq = seq_next; h = h_next; t = t_next;
    count = min(left, nt - t);
    left -= count;
    t_next = 0;
    ++h_next;
    return true;
  }
};

// kExact: a loss gradient E (one bf16 row per window query) takes the place of the attention
// output: T = Vsum E^T needs one product chain instead of two, and the statistics warps form the
// signed sums of g_ij = E^T c_ij instead of the norms (no square roots).
// kShares: the CTA walks a share of all tiles, from unit to unit, else one range of one unit (the caller's rule
// says which).  At a change of unit the query operands are replaced behind the last products that read them:
// about 2.8 thousand cycles in which the statistics warps have nothing, 0.4 of a tile.
template <bool kExact, bool kShares>
__global__ void __launch_bounds__(kBoundThreads, 1)
hessian_stats_tc(const StatsTcArgs a, const RoundTable tab, const __grid_constant__ CUtensorMap tmKp,
                 const __grid_constant__ CUtensorMap tmVp, const __grid_constant__ CUtensorMap tmQ,
                 const __grid_constant__ CUtensorMap tmOhi, const __grid_constant__ CUtensorMap tmOlo) {
  extern __shared__ __align__(1024) uint8_t smem[];
  Misc* misc = reinterpret_cast<Misc*>(smem + kSmemMisc);

  // a group of nqblk CTAs (one per query block, side by side so that they share the tiles in L2) walks the
  // same tiles
  const int qblk = blockIdx.x % a.nqblk, group = blockIdx.x / a.nqblk;
  const int off = tab.off;
  kvs_pdl_launch_dependents();
  Walk walk0 = kShares ? Walk::share(tab, a.Hkv, group, a.tiles_per_group, a.tiles_extra)
                       : Walk::range(tab, group, a.tiles_per_split);
  if (!walk0.next(tab, a.Hkv)) { kvs_pdl_wait(); return; }   // uniform over the CTA
  const int unit0 = tab.s[walk0.seq].b * a.Hkv + walk0.h;
  if (smem_u32(smem) & 1023u) {                        // the swizzled tiles need a 1024-byte aligned base
    kvs_pdl_wait();
    if (threadIdx.x == 0 && a.status_dev) atomicExch(a.status_dev, (int)KVS_ERR_CUDA);
    return;
  }
  // a block of more than 64 queries takes two steps per tile, of half the queries each (to a multiple
  // of 16: eight sequences of 8 K pairs with blocks of 128 and 96 rows, 140 -> 134 us); a smaller block takes
  // one.  The steps go to the two accumulator buffers in turn.
  const int rows = min(kQB, a.M - qblk * kQB);
  const int nh = rows > kQH ? 2 : 1;
  const int qn = ((rows + nh - 1) / nh + 15) & ~15;    // queries of a step

  // (read from one lane, so that the compiler knows the warp index and all that follows from it
  // -- roles, TMEM and barrier addresses -- to be the same in every lane)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    // the staged K rows are free once the last logits are formed, the Vsum rows only after the last
    // T product: each operand is requested again as soon as its own buffer is free
    mbar_init(&misc->kfull, 1);
    mbar_init(&misc->vfull, 1);
    mbar_init(&misc->kfree, kIssuers);     // the issuers' commits
    mbar_init(&misc->vfree, kIssuers);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&misc->tfull[s], kIssuers);
      mbar_init(&misc->tfree[s], kStatWarps);   // statistics warps
    }
    mbar_init(&misc->qfull, 1);
    mbar_init(&misc->qfree, kIssuers);     // a segment's last products: the query operands may be replaced
    mbar_init(&misc->cfull, 1);            // the queries' constants of the segment
    mbar_init(&misc->cfree, kStatWarps);
    mbar_init(&misc->done, kIssuers);      // all products of the CTA
    misc->abort_flag = 0;
    misc->wait_us = (int)a.wait_us;
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&misc->tmem_base, 512);
  // (everything above runs while the kernel before this one may still be draining)
  kvs_pdl_wait();
  // the queries' constants: with one unit they are there before the first tile (a wait for a copy of them in the
  // statistics warps costs 12 registers)
  if (!kShares && threadIdx.x < kQB / 2) {
    reinterpret_cast<float4*>(misc->qconst)[threadIdx.x] =
        reinterpret_cast<const float4*>(a.qc2 + ((size_t)unit0 * a.M_pad + qblk * kQB) * 2)[threadIdx.x];
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, misc->tmem_base, 0);   // (uniform for the compiler too)
  volatile int* abort_flag = &misc->abort_flag;
  // test hook: the producer requests no K tile, so that the waits on them run out
  const bool withhold_k = (a.debug_stall & 2u) != 0;

  // tensor-map coordinates of the pair members: slot = 2 * rho + parity
  const int par_l = off & 1, par_r = par_l ^ 1;
  const int rho_l0 = off >> 1, rho_r0 = (off + 1) >> 1;

  if (warp == 0) {
    // ================================================================ TMA producer
    if (elect_one()) {
      prefetch_tmap(&tmKp); prefetch_tmap(&tmVp); prefetch_tmap(&tmQ); prefetch_tmap(&tmOhi); prefetch_tmap(&tmOlo);
      // K of a tile is free again before its Vsum rows are (the last logits come before the last T
      // product), and the K of the tile after that cannot be free before these Vsum rows have been
      // used: the requests go out in the fixed order K, V, K, V, ... behind blocking (bounded) waits.
      // Every tile is first requested into L2 one tile ahead, so that the load that fills the (single)
      // stage finds it there.  A segment's query operands come after its first K rows.
      uint32_t li = 0, kli = 0, vli = 0, seg = 0, qli = 0, cli = 0;
      bool ok = true;
      Walk w = walk0;
      for (bool more = true; ok && more; more = kShares && w.next(tab, a.Hkv), ++seg) {
        const int b = tab.s[w.seq].b, unit = b * a.Hkv + w.h;
        auto prefetch = [&](int p0, bool v) {
          const CUtensorMap* tm = v ? &tmVp : &tmKp;
          for (int hf = 0; hf < 2; ++hf) {
            tma_prefetch_5d(tm, hf * 64, par_l, rho_l0 + p0, w.h, b);
            tma_prefetch_5d(tm, hf * 64, par_r, rho_r0 + p0, w.h, b);
          }
        };
        auto load_q = [&] {
          if (!mbar_wait(&misc->qfree, (seg & 1) ^ 1, abort_flag)) return false;
          mbar_expect_tx(&misc->qfull, (kExact ? 2 : 3) * kOperand);
          for (int hf = 0; hf < 2; ++hf) {
            tma_load_3d(smem + kSmemQ + hf * kHalf, &tmQ, &misc->qfull, hf * 64, qblk * kQB, unit);
            tma_load_3d(smem + kSmemOhi + hf * kHalf, &tmOhi, &misc->qfull, hf * 64, qblk * kQB, unit);
            if (!kExact) tma_load_3d(smem + kSmemOlo + hf * kHalf, &tmOlo, &misc->qfull, hf * 64, qblk * kQB, unit);
          }
          ++qli;
          return true;
        };
        auto load_c = [&] {
          if (!mbar_wait(&misc->cfree, (seg & 1) ^ 1, abort_flag)) return false;
          mbar_expect_tx(&misc->cfull, sizeof(misc->qconst));
          bulk_load(misc->qconst, a.qc2 + ((size_t)unit * a.M_pad + qblk * kQB) * 2, sizeof(misc->qconst), &misc->cfull);
          ++cli;
          return true;
        };
        if (seg == 0 && (!load_q() || (kShares && !load_c()))) break;
        for (int j = 0; j < w.count; ++j, ++li) {
          const int p0 = (w.t + j) * kPairs;
          if (!mbar_wait(&misc->kfree, (li & 1) ^ 1, abort_flag)) { ok = false; break; }
          if (!withhold_k) {
            mbar_expect_tx(&misc->kfull, 2 * kOperand);
            for (int hf = 0; hf < 2; ++hf) {
              tma_load_5d(smem + kSmemKl + hf * kHalf, &tmKp, &misc->kfull, hf * 64, par_l, rho_l0 + p0, w.h, b);
              tma_load_5d(smem + kSmemKr + hf * kHalf, &tmKp, &misc->kfull, hf * 64, par_r, rho_r0 + p0, w.h, b);
            }
          }
          ++kli;
          if (j + 1 < w.count) prefetch(p0 + kPairs, false);
          if (kShares && j == 0 && seg > 0 && !load_q()) { ok = false; break; }
          if (!mbar_wait(&misc->vfree, (li & 1) ^ 1, abort_flag)) { ok = false; break; }
          mbar_expect_tx(&misc->vfull, 2 * kOperand);
          for (int hf = 0; hf < 2; ++hf) {
            tma_load_5d(smem + kSmemVl + hf * kHalf, &tmVp, &misc->vfull, hf * 64, par_l, rho_l0 + p0, w.h, b);
            tma_load_5d(smem + kSmemVr + hf * kHalf, &tmVp, &misc->vfull, hf * 64, par_r, rho_r0 + p0, w.h, b);
          }
          if (j + 1 < w.count) prefetch(p0 + kPairs, true);
          ++vli;
          if (kShares && j == 0 && seg > 0 && !load_c()) { ok = false; break; }
        }
      }
      misc->k_issued = kli; misc->v_issued = vli; misc->q_issued = qli; misc->c_issued = cli;
      // the last commits, which nobody else waits for, beside the last tile's statistics
      if (!*abort_flag) {
        mbar_drain(&misc->done, 0);
        mbar_drain(&misc->kfree, (kli - 1) & 1);
        mbar_drain(&misc->vfree, (vli - 1) & 1);
        mbar_drain(&misc->qfree, (qli - 1) & 1);
      }
    }
  } else if (warp < kFirstStat) {
    // ================================================================ product issuers
    // warp 1 issues the chains of the left pair members (S_l, T_l), warp 2 those of the right ones
    if (elect_one()) {
      const bool right = warp != 1;
      // descriptors are kept as a constant high word and low words that only need an addition per product
      const uint32_t idesc = idesc_bf16(kPairs, qn);
      const uint32_t dhi = (uint32_t)(smem_desc_sw128(0, 16, 1024) >> 32);
      auto dlo = [&](int off_bytes) { return (uint32_t)smem_desc_sw128(smem_u32(smem + off_bytes), 16, 1024); };
      const uint32_t q_lo = dlo(kSmemQ), ohi_lo = dlo(kSmemOhi), olo_lo = dlo(kSmemOlo);
      const uint32_t k_lo = dlo(right ? kSmemKr : kSmemKl), v_lo = dlo(right ? kSmemVr : kSmemVl);
      bool ok = true;
      uint32_t it = 0, li = 0, seg = 0;
      Walk w = walk0;
      for (bool more = true; ok && more; more = kShares && w.next(tab, a.Hkv), ++seg) {
        if (!mbar_wait(&misc->qfull, seg & 1, abort_flag)) break;
        for (int j = 0; ok && j < w.count; ++j, ++li) {
          if (!mbar_wait(&misc->kfull, li & 1, abort_flag)) { ok = false; break; }
          for (int hq = 0; hq < nh; ++hq, ++it) {
            if (!mbar_wait(&misc->tfree[it & 1], ((it >> 1) & 1) ^ 1, abort_flag)) { ok = false; break; }
            tc_fence_after();
            const uint32_t d0 = tmem + (it & 1) * 256 + (right ? 64u : 0u);
            const uint32_t qrow = (uint32_t)(hq * qn * 128) >> 4;   // rows qn.. of the query-side operands
            const uint32_t qh = q_lo + qrow, oh = ohi_lo + qrow, ol = olo_lo + qrow;
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
              const uint32_t o = ((kk >> 2) * kHalf + (kk & 3) * 32) >> 4;
              if (kk == 0) umma_ss<false>(d0, k_lo, dhi, qh, dhi, idesc);
              else umma_ss<true>(d0, k_lo + o, dhi, qh + o, dhi, idesc);
            }
            if (hq == nh - 1) tc_commit(&misc->kfree);
            if (hq == 0 && !mbar_wait(&misc->vfull, li & 1, abort_flag)) { ok = false; break; }
            // E is one bf16 term, o is two.  Their products take turns: the accumulator is cut at every addition, so that
            // a sum with the lo terms behind the hi terms is cut eight times more at full size (error of N1 against
            // float64 for values around a mean, 1K to 32K slots: 1.62e-5 of the norm, in turn 1.24e-5), and two products
            // in a row read the same rows (8 units of 16 K pairs: 152.3 -> 150.3 us a call).
            constexpr int kTSteps = kExact ? 8 : 16;
#pragma unroll
            for (int kk = 0; kk < kTSteps; ++kk) {
              const int ks = kExact ? kk : kk >> 1;
              const uint32_t o = ((ks >> 2) * kHalf + (ks & 3) * 32) >> 4;
              const uint32_t ob = (kExact || (kk & 1) ? oh : ol) + o;
              if (kk == 0) umma_ss<false>(d0 + 128, v_lo, dhi, ob, dhi, idesc);
              else umma_ss<true>(d0 + 128, v_lo + o, dhi, ob, dhi, idesc);
            }
            tc_commit(&misc->tfull[it & 1]);
          }
          if (!ok) break;
          tc_commit(&misc->vfree);
        }
        if (ok) tc_commit(&misc->qfree);
      }
      tc_commit(&misc->done);                              // (behind a walk that broke off, too)
    }
  } else {
    // ================================================================ statistics warps
    const int grp = (warp - kFirstStat) >> 2;             // its share of the queries of each half
    const int quarter = warp & 3;                         // TMEM lane quarter this warp may read
    const int lane_p = quarter * 32 + lane;               // pair within the tile
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const int nchunk = qn / kChunk;
    uint32_t it = 0, seg = 0;
    bool broken = false;
    Walk w = walk0;
    for (bool more = true; !broken && more; more = kShares && w.next(tab, a.Hkv), ++seg) {
      if constexpr (kShares) w.make_uniform();
      const int unit = tab.s[w.seq].b * a.Hkv + w.h, P = tab.s[w.seq].P;
      const int32_t* Cb = a.counts + (size_t)unit * a.n_max;
      const float4* norms = a.pair_norms + (size_t)unit * a.norm_stride;
      // the partial sums of this (query block, group)
      const size_t sub = (size_t)unit * (a.nqblk * kGroups) + (size_t)qblk * kGroups + grp;
      float4* out4 = a.part4 + sub * a.pair_stride;
      float* out1 = a.part1 + sub * a.pair_stride;
      // norms and counts of the next tile's pair travel while the current tile is reduced
      // (never predicated: the compiler waits for a predicated load where it stands; a lane past the last
      // pair reads that pair's values and its sums are not stored)
      float4 nrm_next;
      int cl_next, cr_next;
      auto fetch = [&](int pn) {
        const int pc = min(pn, P - 1);
        nrm_next = ldg_here(norms + pc);
        cl_next = ldg_here(Cb + off + 2 * pc);
        cr_next = ldg_here(Cb + off + 2 * pc + 1);
      };
      fetch(w.t * kPairs + lane_p);
      if (kShares && !warp_wait(&misc->cfull, seg & 1, abort_flag, lane)) break;
      for (int j = 0; j < w.count; ++j) {
        const int p = (w.t + j) * kPairs + lane_p;          // candidate pair of this thread
        const float4 nrm = nrm_next;
        const float cl = (float)cl_next, cr = (float)cr_next;
        fetch(p + kPairs);
        const float icl = __fdividef(1.f, cl), icr = __fdividef(1.f, cr);   // (counts are small integers)
        const float r2l = nrm.x, r2r = nrm.y, pc = nrm.z;
        const float n2cl = -2.f * cl, n2cr = -2.f * cr, n2il = -2.f * icl, n2ir = -2.f * icr;

        // beta = alpha / c = exp2(scale * s - (max + log2 Z)); sums are scaled by the counts at the end.
        // The arithmetic runs on pairs of neighbouring queries with the packed two-float instructions
        // (fma/add/mul.f32x2): the kernel is as short of issue slots as of special-function slots, and a
        // packed instruction takes one slot for two operations.  Every sum is kept as two lanes.
        float2 sAl = make_float2(0.f, 0.f), sAr = sAl, sN1l = sAl, sN1r = sAl, sN12 = sAl;
        const float2 sc2 = make_float2(a.scale_log2, a.scale_log2), one2 = make_float2(1.f, 1.f);
        const float2 n2cl2 = make_float2(n2cl, n2cl), n2cr2 = make_float2(n2cr, n2cr);
        const float2 n2il2 = make_float2(n2il, n2il), n2ir2 = make_float2(n2ir, n2ir);
        const float2 icl2 = make_float2(icl, icl), icr2 = make_float2(icr, icr);
        const float2 r2l2 = make_float2(r2l, r2l), r2r2 = make_float2(r2r, r2r), pc2 = make_float2(pc, pc);
        const float2 four2 = make_float2(4.f, 4.f), n4il2 = make_float2(2.f * n2il, 2.f * n2il), n4ir2 = make_float2(2.f * n2ir, 2.f * n2ir);
        for (int hq = 0; hq < nh; ++hq, ++it) {
          if (!warp_wait(&misc->tfull[it & 1], (it >> 1) & 1, abort_flag, lane)) { broken = true; break; }
          tc_fence_after();
          const uint32_t col0 = tmem + lane_addr + (it & 1) * 256;
          const float4* qc4 = reinterpret_cast<const float4*>(misc->qconst + hq * (2 * qn));
          // chunks [c_begin, c_end) of every step: 2 / 3 / 3 of the eight of 64 queries.  (Letting the short
          // share go round among the groups measured 1.5 % slower: the group that is done early moves on to
          // the next step and the groups end up staggered, which spreads their serial phases.)
          const int c_begin = (grp * nchunk) / kGroups, c_end = ((grp + 1) * nchunk) / kGroups;
          float buf[4][kChunk];
          // One chunk's loads at a time: the other warps of the scheduler cover their latency.  (With the next
          // chunk's loads in flight, 126 registers instead of 96: 2 % slower.)
#pragma unroll 1
          for (int c = c_begin; c < c_end; ++c) {
            const uint32_t col = col0 + c * kChunk;
            tmem_ld8(col, buf[0]);
            tmem_ld8(col + 64, buf[1]);
            tmem_ld8(col + 128, buf[2]);
            tmem_ld8(col + 192, buf[3]);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < kChunk; i += 2) {
              const float4 cq = qc4[c * (kChunk / 2) + (i >> 1)];           // the two queries' constants (a broadcast read)
              const float2 ncq = make_float2(cq.x, cq.y), hq2 = make_float2(cq.z, cq.w);
              const float2 el = __ffma2_rn(make_float2(buf[0][i], buf[0][i + 1]), sc2, ncq);
              const float2 er = __ffma2_rn(make_float2(buf[1][i], buf[1][i + 1]), sc2, ncq);
              const float2 bl = make_float2(fast_exp2(el.x), fast_exp2(el.y));
              const float2 br = make_float2(fast_exp2(er.x), fast_exp2(er.y));
              const float2 tl = make_float2(buf[2][i], buf[2][i + 1]), tr = make_float2(buf[3][i], buf[3][i + 1]);
              sAl = __fadd2_rn(sAl, bl);
              sAr = __fadd2_rn(sAr, br);
              const float2 al = __ffma2_rn(bl, n2cl2, one2), ar = __ffma2_rn(br, n2cr2, one2);   // 1 - 2 alpha
              if constexpr (kExact) {
                // g11 = alpha (1 - 2 alpha) E^T (vbar_l - o), g12 = -alpha_l alpha_r E^T (vbar_l + vbar_r - 2 o);
                // hq2 holds <E_q, o_q> here (the sign of g12 is applied after the loop)
                const float2 nh2 = make_float2(-hq2.x, -hq2.y);
                const float2 hl = __ffma2_rn(tl, icl2, nh2), hr = __ffma2_rn(tr, icr2, nh2);     // E^T (vbar - o)
                sN1l = __ffma2_rn(__fmul2_rn(bl, al), hl, sN1l);
                sN1r = __ffma2_rn(__fmul2_rn(br, ar), hr, sN1r);
                sN12 = __ffma2_rn(__fmul2_rn(bl, br), __fadd2_rn(hl, hr), sN12);
              } else {
                const float2 gl = make_float2(bl.x * fabsf(al.x), bl.y * fabsf(al.y));          // beta |1 - 2 alpha|
                const float2 gr = make_float2(br.x * fabsf(ar.x), br.y * fabsf(ar.y));
                const float2 dl = __ffma2_rn(tl, n2il2, __fadd2_rn(r2l2, hq2));                  // |vbar_l - o|^2
                const float2 dr = __ffma2_rn(tr, n2ir2, __fadd2_rn(r2r2, hq2));
                sN1l = __ffma2_rn(gl, make_float2(fast_sqrt(fabsf(dl.x)), fast_sqrt(fabsf(dl.y))), sN1l);
                sN1r = __ffma2_rn(gr, make_float2(fast_sqrt(fabsf(dr.x)), fast_sqrt(fabsf(dr.y))), sN1r);
                // |vbar_l + vbar_r - 2 o|^2 = |vbar_l + vbar_r|^2 + 4 |o|^2 - 4 <vbar_l, o> - 4 <vbar_r, o>
                const float2 d12 = __ffma2_rn(tl, n4il2, __ffma2_rn(tr, n4ir2, __ffma2_rn(hq2, four2, pc2)));
                sN12 = __ffma2_rn(__fmul2_rn(bl, br), make_float2(fast_sqrt(fabsf(d12.x)), fast_sqrt(fabsf(d12.y))), sN12);
              }
            }
          }
          tc_fence_before();
          warp_arrive(&misc->tfree[it & 1], lane);                           // the buffer may be overwritten
        }
        if (broken) break;
        // the sums of this (query block, group) for the pair: a later kernel adds the partials in order
        if (p < P) {
          out4[p] = make_float4(cl * (sAl.x + sAl.y), cr * (sAr.x + sAr.y), cl * (sN1l.x + sN1l.y), cr * (sN1r.x + sN1r.y));
          out1[p] = (kExact ? -1.f : 1.f) * cl * cr * (sN12.x + sN12.y);
        }
      }
      if constexpr (kShares) warp_arrive(&misc->cfree, lane);
    }
  }

  // ================================================================== common exit
  // Nothing may be in flight when the CTA leaves: its shared and tensor memory are the next CTA's from then on.  A whole walk
  // has waited for its copies and products; behind one that broke off, in whichever role and after whichever request, any copy
  // and any product may be under way.
  tc_fence_before();
  __syncthreads();
  const bool gave_up = *abort_flag != 0;                   // (no wait is left that could set it)
  if (warp == 1) {
    if (gave_up && lane == 0) mbar_drain(&misc->done, 0);
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (threadIdx.x == 0 && gave_up) {
    const uint32_t nk = misc->k_issued, nv = misc->v_issued, nq = misc->q_issued, nc = misc->c_issued;
    mbar_drain(&misc->done, 0);
    if (nk > 0 && !withhold_k) mbar_drain(&misc->kfull, (nk - 1) & 1);
    if (nv > 0) mbar_drain(&misc->vfull, (nv - 1) & 1);
    if (nq > 0) mbar_drain(&misc->qfull, (nq - 1) & 1);
    if (nc > 0) mbar_drain(&misc->cfull, (nc - 1) & 1);
    if (a.status_dev) atomicExch(a.status_dev, (int)KVS_ERR_TIMEOUT);
  }
}

}  // namespace

cudaError_t kvs_launch_stats_tc(const StatsTcArgs& args, const RoundTable& t, const CUtensorMap& tmKp,
                                const CUtensorMap& tmVp, const CUtensorMap& tmQ, const CUtensorMap& tmOhi,
                                const CUtensorMap& tmOlo, cudaStream_t st) {
  static KvsPerDeviceOnce configured;
  cudaError_t ce = configured.run([] {
    for (auto k : {hessian_stats_tc<false, false>, hessian_stats_tc<false, true>, hessian_stats_tc<true, false>, hessian_stats_tc<true, true>}) {
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  });
  if (ce != cudaSuccess) return ce;
  StatsTcArgs a = args;
  dim3 grid(a.splits * a.nqblk, a.Hkv, t.nseq);
  if (a.splits == 0) {                     // shares: as many groups as fit, one CTA per SM, each with a tile at least
    const int groups = kvs_stats_groups(a.nqblk, a.tiles);
    a.tiles_per_group = a.tiles / groups;
    a.tiles_extra = a.tiles % groups;
    grid = dim3(groups * a.nqblk);
  }
  auto kernel = a.weight_mode == 0 ? (a.splits ? hessian_stats_tc<false, false> : hessian_stats_tc<false, true>)
                                   : (a.splits ? hessian_stats_tc<true, false> : hessian_stats_tc<true, true>);
  return kvs_launch_chained(kernel, grid, dim3(kThreads), kSmemBytes, st, a, t, tmKp, tmVp, tmQ, tmOhi, tmOlo);
}
