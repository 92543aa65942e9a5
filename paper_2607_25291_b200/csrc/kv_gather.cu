// Paged K/V with pages smaller than a key block (Sec. C.1: a logical block may span several physical pages).
//
// The tensor-core kernels fetch a 128-row key tile as one pair of TMA boxes; with b_p < 128 a tile becomes 128 / b_p
// pairs issued by a single thread, and the KAP screen needs at least eight sampled rows per box.  For such pools the
// library first copies the pages of the call's sequences into a dense [B, Hkv, N, d] staging tensor in its scratch
// (one pass over K, or K and V, at HBM speed: 0.1 ms per 268 MB tensor) and runs the dense path on that.
#include <algorithm>

#include "common.cuh"

namespace cosa {
namespace {

// Sixteen lanes take a row (16 bytes each), a warp eight rows at a time: four table look-ups, then four loads in flight a lane.
// grid (row blocks, (batch item, KV head), pools): K and V in one launch.  every: copy only the rows whose token index is a
// multiple of it (KAP reads nothing but its sampled rows; the other rows of the staging tensor stay unwritten).  Bound by memory, or
// by the launch where little is copied.  One chunk a thread and turn, each with its own divisions and look-up, K after V, outside the
// chain of launches: a pass over four prompts of 8K to 16K tokens in 16-token pages took 1 % longer.  kAhead: a warp takes up to eight
// turns, the next one's rows loaded before this one's are stored (K and V of those prompts: the OSK call 660 -> 654 us; KAP's rows,
// an eighth of K's, lose by it).
constexpr int kThreads = 256, kRowsPerWarp = 8;
struct Pools { const uint4* pool[2]; uint4* dense[2]; };
template <bool kAhead>
__global__ void __launch_bounds__(kThreads) gather_pages_kernel(Pools t, KvPaging pg, int batch_heads, int hkv, int n, int every) {
  constexpr int kChunks = kHeadDim * 2 / 16;
  chain_begin();
  const int lane = threadIdx.x & 31, c = lane & 15;
  const uint4* __restrict__ pool = t.pool[blockIdx.z];
  uint4* __restrict__ dense = t.dense[blockIdx.z];
  for (int bg = blockIdx.y; bg < batch_heads; bg += gridDim.y) {
    const int b = bg / hkv, g = bg - b * hkv;
    const int len = pg.seq_lens ? min(n, pg.seq_lens[b]) : n;      // (padding is never read as keys)
    const int rows = (max(len, 0) + every - 1) / every;
    const int32_t* table = pg.table + (long long)b * pg.pages_per_seq;
    constexpr int kSteps = kRowsPerWarp / 2;
    auto load = [&](int r0, uint4 (&w)[kSteps]) {
#pragma unroll
      for (int u = 0; u < kSteps; ++u) {
        const int r = r0 + 2 * u + (lane >> 4), token = r * every;
        if (r < rows)
          w[u] = pool[(((long long)table[token >> pg.page_shift] * hkv + g) * pg.page_size + (token & (pg.page_size - 1))) * kChunks + c];
      }
    };
    auto store = [&](int r0, const uint4 (&w)[kSteps]) {
#pragma unroll
      for (int u = 0; u < kSteps; ++u) {
        const int r = r0 + 2 * u + (lane >> 4);
        if (r < rows) dense[((long long)bg * n + (long long)r * every) * kChunks + c] = w[u];
      }
    };
    const int turn = (int)gridDim.x * (kThreads / 32) * kRowsPerWarp;
    int r0 = (blockIdx.x * (kThreads / 32) + (int)(threadIdx.x >> 5)) * kRowsPerWarp;
    uint4 w[kSteps], next[kSteps];
    if (kAhead && r0 < rows) load(r0, w);
    for (; r0 < rows; r0 += turn) {
      if (!kAhead) load(r0, w);
      if (kAhead && r0 + turn < rows) load(r0 + turn, next);
      store(r0, w);
#pragma unroll
      for (int u = 0; u < kSteps && kAhead; ++u) w[u] = next[u];
    }
  }
}

}  // namespace

cudaError_t launch_gather_pages(const __nv_bfloat16* k_pool, __nv_bfloat16* k_dense, const __nv_bfloat16* v_pool, __nv_bfloat16* v_dense,
                                const KvPaging& pg, int batch, int hkv, int n, int every, cudaStream_t st) {
  if (every < 1 || n % every != 0) return cudaErrorInvalidValue;
  Pools t{};
  t.pool[0] = reinterpret_cast<const uint4*>(k_pool); t.dense[0] = reinterpret_cast<uint4*>(k_dense);
  t.pool[1] = reinterpret_cast<const uint4*>(v_pool); t.dense[1] = reinterpret_cast<uint4*>(v_dense);
  const int per_cta = kThreads / 32 * kRowsPerWarp, heads = batch * hkv, parts = (n / every + per_cta - 1) / per_cta;
  // Turns only where some thousand CTAs are left.  K and V in 16-token pages of 8 KV heads, cold, us with one turn / with the rule's: 4K
  // tokens (one) 16.4, 8K (2 turns) 22.5 / 22.5, 12K (3) 28.7 / 28.7, 16K (4) 35.3 / 34.8, 24K (6) 49.2 / 45.1, 32K (8) 61.4 / 56.8, 128K (8)
  // 221 / 186, four prompts of 10K to 16K (8) 98 / 82.  Twelve gain no more (55 to 184 and 84); two where the rule gives eight lose (225, 106)
  const int turns = v_pool ? (int)std::min<long long>(8, std::max<long long>(1, (long long)parts * heads * 2 / 1024)) : 1;
  const dim3 grid((unsigned)((parts + turns - 1) / turns), (unsigned)(heads < 65535 ? heads : 65535), v_pool ? 2 : 1);
  return launch_chained(turns > 1 ? gather_pages_kernel<true> : gather_pages_kernel<false>, grid, kThreads, 0, st, t, pg, heads, hkv, n, every);
}

}  // namespace cosa
