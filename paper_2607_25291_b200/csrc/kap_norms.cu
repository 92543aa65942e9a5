// KAP fast path, stage 0: the largest squared norm among the sampled key rows of a call (Algorithm A step 2 samples
// every s-th row of Q and K; the screen kernel takes the norms of the sampled query rows itself, from shared memory).
//
// The float32 screen forms its logits on the tensor cores; the rounding error of a logit grows with the size of the
// products it adds up, which |q| |k| bounds (Cauchy-Schwarz).  The thresholds below which the later stages distrust the
// screen -- two block maxima of a row "too close to call", two sorted scores a "near tie" -- therefore follow the
// magnitude of the call's inputs instead of being fixed numbers tuned to one distribution: see screen_error_bound().
#include "common.cuh"

namespace cosa {
namespace {

constexpr int kThreads = 512;
constexpr int kNormRows = 8;

// kNormRows rows in flight per warp, two per load (16 lanes take a row, 16 bytes each); k2part[CTA] = the largest |k_row|^2 among the
// CTA's rows.  (Partial maxima instead of an atomic on one word: nothing has to be cleared first.)  Bound by how many
// loads are in flight: a row is one 256-byte piece per `stride` rows.
__global__ void __launch_bounds__(kThreads) kap_norms_kernel(const __nv_bfloat16* __restrict__ k, KvPaging pg, Strides ks, int batch,
                                                             int hkv, int n, int stride, float* k2part, int32_t* todo, int32_t* slot_taken, int slots) {
  __shared__ float warp_best[kThreads / 32];
  const int lane = threadIdx.x & 31;
  chain_begin();
  if (blockIdx.x == 0 && threadIdx.x < 2) todo[threadIdx.x] = 0;
  for (int t = blockIdx.x * kThreads + threadIdx.x; t < slots; t += gridDim.x * kThreads) slot_taken[t] = 0;   // for the screen
  const long long warp = ((long long)blockIdx.x * kThreads + threadIdx.x) >> 5;
  const long long n_warps = ((long long)gridDim.x * kThreads) >> 5;
  const int ns = n / stride;
  const long long rows = (long long)batch * hkv * ns;
  float best = 0.f;
  for (long long r0 = warp * kNormRows; r0 < rows; r0 += n_warps * kNormRows) {
    uint4 w[kNormRows / 2];
#pragma unroll
    for (int u = 0; u < kNormRows / 2; ++u) {
      const long long r = r0 + 2 * u + (lane >> 4);
      w[u] = make_uint4(0u, 0u, 0u, 0u);
      if (r >= rows) continue;
      const int token = (int)(r % ns) * stride;
      const int bg = (int)(r / ns);
      const int b = bg / hkv;
      if (pg.seq_lens && token >= pg.seq_lens[b]) continue;      // padding past the item's length
      w[u] = reinterpret_cast<const uint4*>(k + kv_off(pg, ks, b, hkv, bg % hkv, token))[lane & 15];
    }
#pragma unroll
    for (int u = 0; u < kNormRows / 2; ++u) {
      const unsigned ws[4] = {w[u].x, w[u].y, w[u].z, w[u].w};
      float s = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float lo = __uint_as_float(ws[q] << 16), hi = __uint_as_float(ws[q] & 0xffff0000u);
        s = fmaf(lo, lo, fmaf(hi, hi, s));
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (s == s) best = fmaxf(best, s);                // (a NaN row is left to the later stages)
    }
  }
  best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, 16));
  if (lane == 0) warp_best[threadIdx.x >> 5] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < kThreads / 32; ++q) best = fmaxf(best, warp_best[q]);
    k2part[blockIdx.x] = best;
  }
}

}  // namespace

cudaError_t launch_kap_norms(KapScreenParams* sp, cudaStream_t st) {
  const long long rows = (long long)sp->batch * sp->hkv * (sp->n / sp->stride);
  const int per_cta = kNormRows * (kThreads / 32);
  long long blocks = (rows + per_cta - 1) / per_cta;
  if (blocks > kNormParts) blocks = kNormParts;
  if (blocks < 1) blocks = 1;
  sp->k2parts = (int)blocks;
  return launch_chained(kap_norms_kernel, dim3((unsigned)blocks), kThreads, 0, st, sp->k, sp->pg, sp->ks, sp->batch, sp->hkv, sp->n,
                        sp->stride, sp->k2part, sp->todo, sp->slot_taken, sp->slots);
}

}  // namespace cosa
