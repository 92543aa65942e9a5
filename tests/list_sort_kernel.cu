// Runs the sort of the screen's lists on its own: a warp a list.  scores [lists, J] (sign: the list's flag); out [lists, 256]: the sorted
// keys; cycles [lists]: clock cycles of the sort.
#include <math.h>

#include "list_sort.cuh"

namespace {

constexpr int kWarps = 4;

template <int PER>
__global__ void sort_lists_kernel(const float* scores, int lists, int J, unsigned long long* out, long long* cycles) {
  __shared__ float score[kWarps][256];
  __shared__ unsigned long long srt[kWarps][256];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, list = blockIdx.x * kWarps + warp;
  if (list >= lists) return;
  unsigned long long key[PER];
  for (int x = 0; x < PER; ++x) {
    const int j = lane + 32 * x;
    const float v = j < J ? scores[(size_t)list * J + j] : 0.f;
    if (j < J) score[warp][j] = v;
    key[x] = j < J ? ((unsigned long long)(__float_as_uint(fabsf(v)) | (v < 0.f ? 0x80000000u : 0u)) << 32) | (0xffffffffu - (unsigned)j) : 0ULL;
  }
  __syncwarp();
  const long long begin = clock64();
  cosa::sort_list<PER>(key, score[warp], J, srt[warp], lane);
  __syncwarp();
  const long long end = clock64();
  for (int t = lane; t < J; t += 32) out[(size_t)list * 256 + t] = srt[warp][t];
  if (lane == 0) cycles[list] = end - begin;
}

}  // namespace

// per: keys a lane (2, 4 or 8; 32 * per >= J).  Returns the CUDA error
extern "C" int sort_lists(const float* scores, int lists, int J, int per, unsigned long long* out, long long* cycles) {
  if (lists < 1 || J < 1 || J > 32 * per) return (int)cudaErrorInvalidValue;
  const int grid = (lists + kWarps - 1) / kWarps;
  if (per == 2) sort_lists_kernel<2><<<grid, 32 * kWarps>>>(scores, lists, J, out, cycles);
  else if (per == 4) sort_lists_kernel<4><<<grid, 32 * kWarps>>>(scores, lists, J, out, cycles);
  else if (per == 8) sort_lists_kernel<8><<<grid, 32 * kWarps>>>(scores, lists, J, out, cycles);
  else return (int)cudaErrorInvalidValue;
  const cudaError_t e = cudaGetLastError();
  return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
