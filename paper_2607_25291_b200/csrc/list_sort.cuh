// The order of a visit list in the screen (kap_screen.cu): a warp sorts up to 256 keys, each a flag, the bits of a score and an id.
#pragma once
#include <stdint.h>

namespace cosa {

// (a whole warp) sorts 32 * PER keys descending (bitonic, in registers); afterwards lane l holds places l * PER and on
template <int PER>
__device__ __forceinline__ void warp_sort_desc(uint32_t (&k)[PER], int lane) {
#pragma unroll
  for (int size = 2; size <= 32 * PER; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride >= PER) {
        const bool larger = ((lane & (size / PER)) == 0) == ((lane & (stride / PER)) == 0);
#pragma unroll
        for (int r = 0; r < PER; ++r) {
          const uint32_t other = __shfl_xor_sync(0xffffffffu, k[r], stride / PER);
          k[r] = larger ? max(k[r], other) : min(k[r], other);
        }
      } else {
#pragma unroll
        for (int r = 0; r < PER; ++r) {
          if (r & stride) continue;
          const bool down = size < PER ? (r & size) == 0 : (lane & (size / PER)) == 0;
          const uint32_t x = max(k[r], k[r | stride]), y = min(k[r], k[r | stride]);
          k[r] = down ? x : y;
          k[r | stride] = down ? y : x;
        }
      }
    }
  }
}
// (a whole warp) puts 32 * PER distinct keys that are all but sorted, held as above, in descending order: neighbours change places
// until none has to, with more than 64 keys kSettleTurns times at most (64 take 33 turns at most).  Returns whether they are in order
constexpr int kSettleTurns = 6;
template <int PER>
__device__ __forceinline__ bool warp_settle_desc(unsigned long long (&k)[PER], int lane) {
  bool swapped;
  int turns = 0;
  do {
    swapped = false;
    auto order = [&](unsigned long long& x, unsigned long long& y) {
      const bool swap = y > x;
      const unsigned long long t = x;
      x = swap ? y : x;
      y = swap ? t : y;
      swapped = swapped || swap;
    };
#pragma unroll
    for (int r = 0; r + 1 < PER; r += 2) order(k[r], k[r + 1]);
#pragma unroll
    for (int r = 1; r + 1 < PER; r += 2) order(k[r], k[r + 1]);
    // the last key of a lane and the first of the next
    const unsigned long long next = __shfl_down_sync(0xffffffffu, k[0], 1), before = __shfl_up_sync(0xffffffffu, k[PER - 1], 1);
    if (lane < 31 && next > k[PER - 1]) { k[PER - 1] = next; swapped = true; }
    if (lane > 0 && before < k[0]) { k[0] = before; swapped = true; }
    swapped = __any_sync(0xffffffffu, swapped);
  } while (swapped && (PER == 2 || ++turns < kSettleTurns));
  return !swapped;
}

// (a whole warp) sorts the J keys of a list descending into srt[].  key[x]: that of id lane + 32 x, 0 from J on: bit 63 its flag, bits 62
// to 32 its score's, the low word 0xffffffff - id.  score[id]: the scores (their sign is not looked at).
// Sorted by words of a flag, the leading bits of the score and the id, which is a third of the work of sorting whole keys; what that
// leaves out of order is close together and settled after, in a turn or two.  Scores of one word that rise with their ids
// (near-duplicate blocks) lie in reverse and would take half as many turns as there are, 184 cycles each; so what a few turns do not settle
// is sorted once more, by words of the run of equal leading bits, the score's last byte and the id.  Cycles of a warp for 256 scores far
// apart / of one word: 1,850 / 5,200 (settled to the end: 1,780 / 25,300; whole keys sorted in shared memory instead: 18,700).  Stage 1 with
// seven of eight blocks alike, rising, by sorting whole keys from the first / by settling to the end / so: 201 blocks 139 / 160 / 133 us,
// 256 blocks 366 / 401 / 354.
// (Ids are below 256.  A word of 0 is no key, or the last of 256)
template <int PER>
__device__ __forceinline__ void sort_list(unsigned long long (&key)[PER], const float* score, int J, unsigned long long* srt, int lane) {
  static_assert(32 * PER <= 256, "an id is a byte");
  uint32_t word[PER];
  auto sort = [&]() {
    warp_sort_desc<PER>(word, lane);
#pragma unroll
    for (int x = 0; x < PER; ++x) {
      const uint32_t j = 0xffu - (word[x] & 0xffu);
      key[x] = lane * PER + x < J ? ((unsigned long long)((word[x] & 0x80000000u) | __float_as_uint(fabsf(score[j]))) << 32) | (0xffffffffu - j) : 0ULL;
    }
  };
#pragma unroll
  for (int x = 0; x < PER; ++x) word[x] = ((uint32_t)(key[x] >> 32) & 0xffffff00u) | (lane + 32 * x < J ? 0xffu - (uint32_t)(lane + 32 * x) : 0u);
  sort();
  const bool in_order = warp_settle_desc<PER>(key, lane);
  if (PER > 2 && !in_order) {
    // place where the run of a key's leading bits begins (keys have changed places within their runs only): the last begin so far
    const uint32_t before = __shfl_up_sync(0xffffffffu, (uint32_t)(key[PER - 1] >> 40), 1);
    int begin[PER], last = 0;
#pragma unroll
    for (int x = 0; x < PER; ++x) {
      const uint32_t lead = (uint32_t)(key[x] >> 40);
      if (lead != (x > 0 ? (uint32_t)(key[x > 0 ? x - 1 : 0] >> 40) : before)) last = lane * PER + x;   // (lane 0's first: 0 either way)
      begin[x] = last;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int of = __shfl_up_sync(0xffffffffu, last, o);
      if (lane >= o) last = max(last, of);
    }
    last = __shfl_up_sync(0xffffffffu, last, 1);
#pragma unroll
    for (int x = 0; x < PER; ++x) {
      const uint32_t run = 255u - (uint32_t)(lane > 0 ? max(begin[x], last) : begin[x]);
      word[x] = ((uint32_t)(key[x] >> 32) & 0x80000000u) | (run << 16) | ((uint32_t)(key[x] >> 24) & 0xff00u) | ((uint32_t)key[x] & 0xffu);
    }
    sort();
  }
#pragma unroll
  for (int x = 0; x < PER; ++x) srt[lane * PER + x] = key[x];
}

}  // namespace cosa
