// Merge of the selected adjacent pairs and stable in-place compaction of the cache.
//
// A tile is 64 consecutive slots starting at the first candidate slot (32 candidate pairs;
// tiles past the last pair only shift the protected tail).  CTAs are persistent: within one
// (sequence, KV head) they take tiles by ticket.  A producer warp takes the ticket, streams
// the tile's K and Vsum rows into a three-stage shared-memory ring with bulk asynchronous
// copies, and stages the tile's decision (mask bits, weights, counts, merged pairs before the
// tile).  Eight consumer warps read the rows into registers, free the stage, form the merged
// rows
//   K*    = bf16( K_right + w (K_left - K_right) )        [Eq. kstar_final, weight form]
//   Vsum* = bf16( Vsum_left + Vsum_right ),  c* = c_left + c_right   [v* = v_m + v_{m+1}]
// wait until the tile may be stored, that is until every earlier tile whose source rows it overwrites has loaded, and store the
// surviving rows at
//   new slot = old slot - (merged pairs before it).
// Where several CTAs handle tiles of a unit, a publisher warp says that a tile has loaded, as soon as its copies have landed or
// a few tiles later.
// A gate warp waits (bounded) for the other tiles in place of all consumers and opens a tile for them: it is stored by
// all of them or, behind a wait that ran out, by none.
// Tickets make the wait safe: a tile only waits for tiles of its unit with smaller tickets, which were taken before its own.
// Every CTA handles its tiles, of one unit or of several, in the order in which it took them, and publishes one without waiting
// for anything but tiles that it took before, so that of all tiles not yet published the one taken first never waits.
// Bound by HBM in long units, by the chain of ticket, copies, flags and stores in short ones.  8 units of 2048 tiles 152 us a
// launch (events), nine rounds of 8 units from 512 tiles on 185, five of 8 units from 64 on 67; with barriers of all consumers
// around every wait, and flags set and looked at by consumers, 185, 248 and 73.
#include "kvs_internal.h"
#include "kvs_sm100.cuh"

using namespace sm100;

namespace {

__device__ __forceinline__ uint32_t merge_k2(uint32_t l, uint32_t r, float w) {
  const float l0 = bf16lo(l), l1 = bf16hi(l), r0 = bf16lo(r), r1 = bf16hi(r);
  const float a = fmaf(w, l0 - r0, r0), b = fmaf(w, l1 - r1, r1);
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ uint32_t add_v2(uint32_t l, uint32_t r) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(bf16lo(l) + bf16lo(r), bf16hi(l) + bf16hi(r));
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ uint4 merge_k8(uint4 l, uint4 r, float w) {
  return make_uint4(merge_k2(l.x, r.x, w), merge_k2(l.y, r.y, w), merge_k2(l.z, r.z, w),
                    merge_k2(l.w, r.w, w));
}
__device__ __forceinline__ uint4 add_v8(uint4 l, uint4 r) {
  return make_uint4(add_v2(l.x, r.x), add_v2(l.y, r.y), add_v2(l.z, r.z), add_v2(l.w, r.w));
}

constexpr int kStages = 3;
constexpr int kRowBytes = KVS_D * 2;                       // one bf16 row
constexpr int kOperandBytes = KVS_CTILE * kRowBytes;       // 16 KB: the K (or Vsum) rows of a tile
constexpr int kStageBytes = 2 * kOperandBytes;
constexpr int kConsumers = 256;
constexpr int kProducer = kConsumers / 32, kPublisher = kProducer + 1, kGate = kProducer + 2;   // warps
constexpr int kThreads = kConsumers + 96;
// Barriers of the gate's verdicts: a consumer arrives on `empty` of a tile before it waits for the verdict, and is past the
// verdict on tile k when it arrives for tile k + kStages, without which tile k + 2 kStages has no stage.
constexpr int kOpen = 2 * kStages;
constexpr uint32_t kNever = 0xffffffffu;

struct TileMeta {
  int32_t tile;                  // -1: no more tiles
  int32_t E0;                    // merged pairs before the tile
  uint32_t selbits;              // bit i: pair i of the tile is merged
  int32_t seq, h;                // the tile's unit: entry of the launch table, KV head
  float w[32];
  int32_t cnt[KVS_CTILE];
};
struct Shared {
  uint64_t full[kStages], meta_full[kStages], empty[kStages];
  uint64_t open[kOpen];          // the rows of the tile may be stored
  int abort_flag, wait_us;       // (adjacent: the bounded waits read both through one pointer)
  uint32_t closed;               // written by the gate only: it has opened this many of the CTA's tiles and will open no more
  TileMeta meta[kStages];
};
constexpr int kSmemBytes = kStages * kStageBytes + (int)sizeof(Shared);

// The "tile loaded" flags order a read before a write: the copies of a tile's rows and counts, complete when the flag is set,
// before the stores that overwrite them in another CTA.  Release and acquire are what the memory model has for that.  The
// acquire is free in the gate, the release is not: with relaxed flags 8 units of 256 tiles take 22.5 us a launch and
// so 24.5, of 2048 149 and 152, 128 of 256 300 and 309, all rounds of a ragged batch of 4 K to 64 K slots 927 and 977.
// They are looked at with an atomic, which goes to the one place where the line lives.  A load leaves copies of a line that is
// about to be written in the caches in between: a CTA that looked a little too early saw the flag 2 us late (with a release for
// every tile, 8 units of 256 tiles with loads 34.4 us, with atomics 23.2; 64 units of 24 tiles 23.0 and 20.9).
__device__ __forceinline__ uint32_t see_flag(uint32_t* p) {
  uint32_t v;
  asm volatile("atom.acquire.gpu.global.or.b32 %0, [%1], 0;" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_flag(uint32_t* p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// One lane waits, the warp follows.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int lane) {
  int ok = 1;
  if (lane == 0) ok = mbar_wait(bar, parity, abort_flag) ? 1 : 0;
  ok = __shfl_sync(0xffffffffu, ok, 0);
  __syncwarp();
  return ok != 0;
}

// The consumers' waits, which end with the phase or with the gate: they never give up on a tile that the gate has opened or
// may still open.  The gate itself gives up on a tile after three time limits at the most (decision, flags, copies);
// far beyond that the wait ends all the same.
__device__ __forceinline__ uint32_t ld_closed(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ void st_closed(uint32_t* p, uint32_t v) {
  asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ bool follow(uint64_t* bar, uint32_t parity, Shared* sh, uint32_t k, int lane) {
  int ok = 1;
  if (lane == 0 && !mbar_try_wait(bar, parity)) {
    const uint64_t since = globaltimer_ns();
    while (!mbar_try_wait_hint(bar, parity, 10000u)) {
      const bool late = globaltimer_ns() - since > (uint64_t)(uint32_t)sh->wait_us * 8000ull + 100000000ull;
      if (late) *(volatile int*)&sh->abort_flag = 1;
      if (late || ld_closed(&sh->closed) <= k) { ok = 0; break; }
    }
  }
  ok = __shfl_sync(0xffffffffu, ok, 0);
  __syncwarp();
  return ok != 0;
}

// Persistent CTAs per unit: the 2 x 148 CTAs that fit the GPU are shared out in proportion to the
// units' tile counts (a ragged batch would otherwise wait for its longest sequence, which would
// have no more CTAs than the shortest), at least one and at most one per tile.
__host__ __device__ inline int ctas_of_unit(int unit_tiles, long long all_tiles, bool share) {
  if (unit_tiles <= 0) return 0;
  // rounded down: all of them are resident at once; rounded up where a CTA that has no tile left goes on with other units
  long long c = all_tiles > 0 ? (2LL * 148 * unit_tiles + (share ? all_tiles - 1 : 0)) / all_tiles : 1;
  if (c < 1) c = 1;
  if (c > unit_tiles) c = unit_tiles;
  return (int)c;
}
__host__ __device__ inline int tiles_of(int n, int off) { return n > off ? (n - off + KVS_CTILE - 1) / KVS_CTILE : 0; }

__global__ void __launch_bounds__(kThreads, 2)
merge_compact_kernel(const CompactArgs a, const RoundTable tab) {
  extern __shared__ __align__(128) uint8_t smem[];
  Shared* sh = reinterpret_cast<Shared*>(smem + kStages * kStageBytes);
  kvs_pdl_launch_dependents();
  const int seq = blockIdx.z;
  const SeqRound sr = tab.s[seq];
  const int n = sr.n;
  const int h = blockIdx.y;
  const int unit = sr.b * a.c.Hkv + h;
  const int off = tab.off;
  const int ntiles = tiles_of(n, off);
  long long all_tiles = 0;
  for (int i = 0; i < tab.nseq; ++i) all_tiles += tiles_of(tab.s[i].n, off);
  const bool share = a.share != 0;
  const int unit_ctas = ctas_of_unit(ntiles, all_tiles * a.c.Hkv, share);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool ordered = share || unit_ctas > 1;             // others handle tiles of the unit, too
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sh->full[s], 1);
      mbar_init(&sh->meta_full[s], 1);
      mbar_init(&sh->empty[s], kConsumers / 32 + 1 + (ordered ? 1 : 0));
    }
    for (int s = 0; s < kOpen; ++s) mbar_init(&sh->open[s], 1);
    sh->abort_flag = 0;
    sh->closed = kNever;
    sh->wait_us = (int)a.wait_us;
    mbar_fence_init();
  }
  __syncthreads();
  // (everything above runs while the kernel before this one may still be draining)
  kvs_pdl_wait();
  if (n <= 0) return;
  if (ntiles == 0) {
    // a unit that ends inside the protected prefix has nothing to move; its slot map is the identity
    if (a.new_index && blockIdx.x == 0) {
      int32_t* ni = a.new_index + (size_t)unit * a.c.n_max;
      for (int j = threadIdx.x; j < n; j += kThreads) ni[j] = j;
    }
    return;
  }
  if ((int)blockIdx.x >= unit_ctas) return;                // this unit's share of the CTAs is smaller
  volatile int* abort_flag = &sh->abort_flag;

  if (warp == kProducer) {
    // ================================================================ producer warp
    // the unit whose tiles it takes: its own, then (share) the one that has the most left
    int cs = seq, ch = h, cu = unit, cn = n, cP = sr.P, ct = ntiles;
    uint32_t next_ticket = 0;
    bool ahead = false;              // next_ticket is taken already
    int issued = 0;                  // tiles whose copies were requested
    for (int k = 0;; ++k) {
      const int s = k % kStages;
      const uint32_t ph = (uint32_t)(k / kStages) & 1u;
      if (!warp_wait(&sh->empty[s], ph ^ 1u, abort_flag, lane)) break;
      int t;
      for (;;) {
        if (!ahead && lane == 0) next_ticket = atomicAdd(&a.tickets[cu], 1u);
        ahead = false;
        t = (int)__shfl_sync(0xffffffffu, next_ticket, 0);
        if (t < ct || !share) break;
        // (a count that is out of date costs a look more, no tile: the ticket decides)
        int left = 0, at = 0;
        for (int i = lane; i < tab.nseq * a.c.Hkv; i += 32) {
          const int q = i / a.c.Hkv, nt = tiles_of(tab.s[q].n, off);
          const int l = nt - (int)*(volatile const uint32_t*)&a.tickets[tab.s[q].b * a.c.Hkv + (i - q * a.c.Hkv)];
          if (l > left) { left = l; at = i; }
        }
        const int most = __reduce_max_sync(0xffffffffu, left);
        if (most <= 0) break;
        at = __shfl_sync(0xffffffffu, at, __ffs((int)__ballot_sync(0xffffffffu, left == most)) - 1);
        cs = at / a.c.Hkv; ch = at - cs * a.c.Hkv;
        cu = tab.s[cs].b * a.c.Hkv + ch; cn = tab.s[cs].n; cP = tab.s[cs].P; ct = tiles_of(cn, off);
      }
      TileMeta* m = &sh->meta[s];
      if (t >= ct) {
        if (lane == 0) { m->tile = -1; mbar_arrive(&sh->meta_full[s]); }
        break;
      }
      const uint8_t* mask = a.mask + (size_t)cu * a.pair_stride;
      const float* wl = a.w + (size_t)cu * a.pair_stride;
      const __nv_bfloat16* Kb = a.c.K + tab.s[cs].b * a.c.ksb + ch * a.c.ksh;
      const __nv_bfloat16* Vb = a.c.V + tab.s[cs].b * a.c.vsb + ch * a.c.vsh;
      const int32_t* Cb = a.c.counts + (size_t)cu * a.c.n_max;
      if (lane == 0) next_ticket = atomicAdd(&a.tickets[cu], 1u);   // its latency hides behind this tile
      ahead = true;
      const int j0 = off + KVS_CTILE * t;
      const int rows = min(KVS_CTILE, cn - j0);
      uint8_t* sk = smem + s * kStageBytes;
      uint8_t* sv = sk + kOperandBytes;
      if (lane == 0) mbar_expect_tx(&sh->full[s], (uint32_t)rows * 2u * kRowBytes);
      issued = k + 1;
      __syncwarp();
      if (a.c.kst == KVS_D && a.c.vst == KVS_D) {
        if (lane == 0) bulk_load(sk, Kb + (int64_t)j0 * KVS_D, (uint32_t)rows * kRowBytes, &sh->full[s]);
        if (lane == 1) bulk_load(sv, Vb + (int64_t)j0 * KVS_D, (uint32_t)rows * kRowBytes, &sh->full[s]);
      } else {
        for (int r = lane; r < rows; r += 32) {
          bulk_load(sk + r * kRowBytes, Kb + (int64_t)(j0 + r) * a.c.kst, kRowBytes, &sh->full[s]);
          bulk_load(sv + r * kRowBytes, Vb + (int64_t)(j0 + r) * a.c.vst, kRowBytes, &sh->full[s]);
        }
      }
      // the tile's decision (all of it requested before the first of it is used)
      const int pp = 32 * t + lane;
      const int32_t E0 = a.tile_prefix[(size_t)cu * a.tile_stride + t];
      const int32_t c0 = Cb[j0 + min(lane, rows - 1)], c1 = Cb[j0 + min(lane + 32, rows - 1)];   // (those past the end are not used)
      uint8_t chosen = 0;
      float weight = 0.5f;
      if (32 * t < cP) {
        chosen = mask[min(pp, cP - 1)];
        weight = wl[min(pp, cP - 1)];
      }
      m->w[lane] = weight;
      m->cnt[lane] = c0;
      m->cnt[lane + 32] = c1;
      const uint32_t bits = __ballot_sync(0xffffffffu, pp < cP && chosen != 0);
      if (lane == 0) {
        m->selbits = bits;
        m->E0 = E0;
        m->seq = cs;
        m->h = ch;
        m->tile = t;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->meta_full[s]);
    }
    // No copy may be in flight when the CTA leaves, whoever gave up and when.
    if (lane == 0)
      for (int kk = max(0, issued - kStages); kk < issued; ++kk) mbar_drain(&sh->full[kk % kStages], (uint32_t)(kk / kStages) & 1u);
  } else if (warp == kPublisher) {
    // ================================================================ publisher
    // (up to two tiles before the consumers get to them; a publisher that also waited for the other tiles' flags was late with
    // its next tile: nine rounds of 8 units from 512 tiles on 220 us, so 187)
    // A tile that nobody overwrites soon -- the first that does so follows E0 slots later -- waits for up to two more tiles, so that
    // one release serves three: 128 units of 256 tiles 331 -> 309 us a launch, 8 of 2048 158 -> 152.  With no more
    // tiles than stages, the last one's stage comes free with tiles taken before the first.
    uint32_t* mine = nullptr;        // of lane i: the i-th flag to be set
    int due = 0;
    for (int k = 0; ordered; ++k) {
      const int s = k % kStages;
      const uint32_t ph = (uint32_t)(k / kStages) & 1u;
      if (!warp_wait(&sh->meta_full[s], ph, abort_flag, lane)) break;
      const TileMeta* m = &sh->meta[s];
      const bool more = m->tile >= 0;
      bool in_time = false;
      if (more) {
        if (lane == due) mine = a.flags + (size_t)(tab.s[m->seq].b * a.c.Hkv + m->h) * a.tile_stride + m->tile;
        in_time = m->E0 >= 3 * unit_ctas * KVS_CTILE;
        if (!warp_wait(&sh->full[s], ph, abort_flag, lane)) break;
        if (lane == 0) mbar_arrive(&sh->empty[s]);
        ++due;
      }
      if (!in_time || due == kStages) {
        // (test hook: with bit 2 of debug_stall the flags stay unset, so that the waits on them run out)
        if (lane < due && !(a.debug_stall & 4u)) st_flag(mine, a.epoch);
        due = 0;
      }
      if (!more) break;
    }
  } else if (warp == kGate) {
    // ================================================================ gate
    uint32_t k = 0;
    bool shut = false;
    for (;; ++k) {
      const int s = (int)(k % kStages);
      const uint32_t ph = (k / kStages) & 1u;
      shut = !warp_wait(&sh->meta_full[s], ph, abort_flag, lane);
      if (shut) break;
      const TileMeta* m = &sh->meta[s];
      const int t = m->tile, E0 = m->E0;
      if (t < 0) break;
      uint32_t* flags = a.flags + (size_t)(tab.s[m->seq].b * a.c.Hkv + m->h) * a.tile_stride;
      if (ordered && E0 > 0) {
        // The tile's rows land in [j0 - E0, j0 - E0 + 64): those are source rows of at most two earlier tiles (and of
        // this tile itself), which must have been read before they are overwritten; a CTA that owns the whole unit has
        // read them itself, in order.
        const int before = (KVS_CTILE * t - E0) / KVS_CTILE + lane;
        shut = lane < 2 && before < t;
        int spins = 0;
        const uint64_t since = globaltimer_ns();
        while (shut && (shut = see_flag(flags + before) < a.epoch)) {
          const bool late = (++spins & 255) == 0 && globaltimer_ns() - since > (uint64_t)(uint32_t)sh->wait_us * 1000ull;
          if (late || spins > KVS_SPIN_LIMIT || *abort_flag) { *abort_flag = 1; break; }
        }
        shut = __any_sync(0xffffffffu, shut);
        if (shut) break;
      }
      shut = !warp_wait(&sh->full[s], ph, abort_flag, lane);
      if (shut) break;
      if (lane == 0) {
        mbar_arrive(&sh->empty[s]);
        mbar_arrive(&sh->open[k % kOpen]);
      }
    }
    if (lane == 0 && shut) st_closed(&sh->closed, k);
  } else {
    // ================================================================ consumer warps
    const int i = tid >> 3;          // pair in tile
    const int c0 = tid & 7;          // chunks c0 and c0 + 8 (16 bytes each)
    // (no warp waits for another one: barriers of all eight around the waits were the kernel's largest stall)
    for (int k = 0;; ++k) {
      const int s = k % kStages;
      const uint32_t ph = (uint32_t)(k / kStages) & 1u;
      if (!follow(&sh->meta_full[s], ph, sh, k, lane)) break;
      const TileMeta* m = &sh->meta[s];
      const int t = m->tile;
      if (t < 0) break;
      if (!follow(&sh->full[s], ph, sh, k, lane)) break;
      const int ts = m->seq, th = m->h;                   // (the tile's unit)
      const int n = tab.s[ts].n, unit = tab.s[ts].b * a.c.Hkv + th;
      __nv_bfloat16* Kb = a.c.K + tab.s[ts].b * a.c.ksb + th * a.c.ksh;
      __nv_bfloat16* Vb = a.c.V + tab.s[ts].b * a.c.vsb + th * a.c.vsh;
      int32_t* Cb = a.c.counts + (size_t)unit * a.c.n_max;
      const int j0 = off + KVS_CTILE * t;
      const int jl = j0 + 2 * i, jr = jl + 1;
      const bool okl = jl < n, okr = jr < n;
      const uint8_t* sk = smem + s * kStageBytes;
      const uint8_t* sv = sk + kOperandBytes;
      uint4 kl[2], kr[2], vl[2], vr[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int ob = (c0 + 8 * u) * 16;
        kl[u] = *reinterpret_cast<const uint4*>(sk + (2 * i) * kRowBytes + ob);
        kr[u] = *reinterpret_cast<const uint4*>(sk + (2 * i + 1) * kRowBytes + ob);
        vl[u] = *reinterpret_cast<const uint4*>(sv + (2 * i) * kRowBytes + ob);
        vr[u] = *reinterpret_cast<const uint4*>(sv + (2 * i + 1) * kRowBytes + ob);
      }
      const uint32_t selbits = m->selbits;
      const int E0 = m->E0;
      const float w = m->w[i];
      int32_t cl = m->cnt[2 * i], cr = m->cnt[2 * i + 1];
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->empty[s]);          // the stage may be refilled

      const bool sel = (selbits >> i) & 1u;
      const int e = __popc(selbits & ((1u << i) - 1u));
      const int dl = jl - E0 - e;
      const int dr = jr - E0 - e;      // used only when !sel
      if (sel) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          kl[u] = merge_k8(kl[u], kr[u], w);
          vl[u] = add_v8(vl[u], vr[u]);
        }
        cl += cr;
      }
      const int moved = E0 + __popc(selbits);
      if (!follow(&sh->open[k % kOpen], (uint32_t)(k / kOpen) & 1u, sh, k, lane)) break;
      if (moved != 0) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int ch = (c0 + 8 * u) * 8;
          if (okl && (sel || dl != jl)) {
            *reinterpret_cast<uint4*>(Kb + (int64_t)dl * a.c.kst + ch) = kl[u];
            *reinterpret_cast<uint4*>(Vb + (int64_t)dl * a.c.vst + ch) = vl[u];
          }
          if (okr && !sel && dr != jr) {
            *reinterpret_cast<uint4*>(Kb + (int64_t)dr * a.c.kst + ch) = kr[u];
            *reinterpret_cast<uint4*>(Vb + (int64_t)dr * a.c.vst + ch) = vr[u];
          }
        }
        if (c0 == 0) {
          if (okl) Cb[dl] = cl;
          if (okr && !sel) Cb[dr] = cr;
        }
      }
      if (a.new_index && c0 == 0) {
        int32_t* ni = a.new_index + (size_t)unit * a.c.n_max;
        if (okl) ni[jl] = dl;
        if (okr) ni[jr] = sel ? dl : dr;
      }
      if (a.new_index && t == 0) {
        int32_t* ni = a.new_index + (size_t)unit * a.c.n_max;
        for (int j = tid; j < off && j < n; j += kConsumers) ni[j] = j;
      }
    }
  }
  __syncthreads();
  if (tid == 0 && sh->abort_flag && a.status_dev) atomicExch(a.status_dev, (int)KVS_ERR_TIMEOUT);
}

}  // namespace

// Persistent CTAs, two per SM over all units of the launch, in proportion to the units' lengths; the grid is as wide as the
// longest unit's part, the CTAs beyond a unit's part leave at once.
// Where the rounding of the parts, or one CTA to each of many units, leaves a unit with a quarter more tiles a CTA than
// the average, CTAs that are done go on with the unit that has most left.  All units then need the flags, and a CTA
// changes its unit for few tiles at a time where units are short, so only from 40 tiles of the busiest CTA on.  Us a launch
// without and with the others' help: 160 units of 63 tiles 130 and 109, 256 of 65 to 124 256 and 234, 128 of 72 to 125 160 and 128, 64 of 265 to
// 444 219 and 213; but 192 of 17 90 and 141, 256 of 20 to 38 86 and 109, of 11 to 37 80 and 93, 128 of 11 to 36 37 and 40; and
// less than a quarter above the average 80 of 63 64 and 62, 96 of 67 73 and 76, 32 of 134 to 376 93 and 96.
int kvs_detail_compact_shares(const int32_t* tiles, int32_t nseq, int32_t Hkv, int32_t* per_unit) {
  long long all_tiles = 0;
  for (int i = 0; i < nseq; ++i) all_tiles += tiles[i];
  all_tiles *= Hkv;
  for (int share = 0;; ++share) {
    double worst = 0.;                                     // tiles of the CTA that has most of them
    *per_unit = 1;
    for (int i = 0; i < nseq; ++i) {
      const int c = ctas_of_unit(tiles[i], all_tiles, share != 0);
      if (c > *per_unit) *per_unit = c;
      if (c > 0 && (double)tiles[i] / c > worst) worst = (double)tiles[i] / c;
    }
    if (share || !(worst >= 40. && worst * (2 * 148) > 1.25 * (double)all_tiles)) return share;
  }
}

cudaError_t kvs_launch_compact(const CompactArgs& a, const RoundTable& t, cudaStream_t st) {
  static KvsPerDeviceOnce configured;
  cudaError_t ce = configured.run([] {
    return cudaFuncSetAttribute(merge_compact_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  });
  if (ce != cudaSuccess) return ce;
  int nmax = 0;
  for (int i = 0; i < t.nseq; ++i) nmax = nmax > t.s[i].n ? nmax : t.s[i].n;
  const int ntiles = (nmax - t.off + KVS_CTILE - 1) / KVS_CTILE;
  // (units that end inside the protected prefix still get their identity slot map)
  if (nmax <= 0 || (ntiles <= 0 && !a.new_index)) return cudaSuccess;
  CompactArgs args = a;
  int32_t tiles[KVS_SEQ_CHUNK], per_unit = 1;
  for (int i = 0; i < t.nseq; ++i) tiles[i] = tiles_of(t.s[i].n, t.off);
  args.share = kvs_detail_compact_shares(tiles, t.nseq, a.c.Hkv, &per_unit);
  dim3 grid(per_unit, a.c.Hkv, t.nseq);
  return kvs_launch_chained(merge_compact_kernel, grid, dim3(kThreads), kSmemBytes, st, args, t);
}
