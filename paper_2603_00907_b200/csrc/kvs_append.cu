// Appending a chunk of fresh tokens to the caches of a layer (the first half of a streaming step).
//
// Row r of the chunk of (sequence b, KV head h) goes to slot n_b + r of that unit, n_b being the
// slots in use; its count becomes 1 and its value sum is its value.  Plain copies, bound by bytes in flight: sixteen
// threads take a row, and a thread requests its 16 bytes of two rows of keys and of two of values before it stores
// the first of them.  256 units of 512 rows (134 MB moved), events around the launch: 30-32 us with one warp per row and
// one request per thread, which took four times the CTAs, 24 us so.
#include "kvs_internal.h"

namespace {

constexpr int kThreads = 256;
constexpr int kStep = kThreads / 16;       // rows side by side
constexpr int kRows = 2 * kStep;           // rows of the chunk that a CTA copies

__global__ void __launch_bounds__(kThreads)
append_chunk_kernel(const AppendArgs a, const RoundTable tab) {
  kvs_pdl_launch_dependents();
  kvs_pdl_wait();
  const SeqRound sr = tab.s[blockIdx.z];
  const int unit = sr.b * a.c.Hkv + (int)blockIdx.y;
  const int r0 = blockIdx.x * kRows + ((int)threadIdx.x >> 4), c = threadIdx.x & 15;
  const int rows = min(a.chunk_len, a.c.n_max - sr.n);     // (the host has checked that all fit)
  const size_t src = ((size_t)unit * a.chunk_len + r0) * (KVS_D / 8) + c;
  uint4 k[2], v[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    if (r0 + i * kStep >= rows) continue;
    k[i] = reinterpret_cast<const uint4*>(a.chunk_k)[src + (size_t)i * kStep * (KVS_D / 8)];
    v[i] = reinterpret_cast<const uint4*>(a.chunk_v)[src + (size_t)i * kStep * (KVS_D / 8)];
  }
  __nv_bfloat16* K = a.c.K + sr.b * a.c.ksb + blockIdx.y * a.c.ksh + 8 * c;
  __nv_bfloat16* V = a.c.V + sr.b * a.c.vsb + blockIdx.y * a.c.vsh + 8 * c;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = r0 + i * kStep;
    if (r >= rows) continue;
    *reinterpret_cast<uint4*>(K + (int64_t)(sr.n + r) * a.c.kst) = k[i];
    *reinterpret_cast<uint4*>(V + (int64_t)(sr.n + r) * a.c.vst) = v[i];
    if (c == 0) a.c.counts[(size_t)unit * a.c.n_max + sr.n + r] = 1;
  }
}

}  // namespace

cudaError_t kvs_launch_append(const AppendArgs& a, const RoundTable& t, cudaStream_t st) {
  dim3 grid((a.chunk_len + kRows - 1) / kRows, a.c.Hkv, t.nseq);
  return kvs_launch_chained(append_chunk_kernel, grid, dim3(kThreads), 0, st, a, t);
}
