// KAP fast path, stage B: flag-grouped sort and retained prefix (Eqs. 13-14; Algorithm A step 5;
// budget count or Top-p, text after Eq. 13)
// on the float32 screen, with a double-precision recount of every decision a rounding error
// could change.
//
// One CTA of four warps per (query head, query block): its time is a chain of short steps, and what counts is how many lists an SM
// has in work: ten, where eight warps a list and the recount's register needs allowed six (this kernel and the recount: 372 ->
// 193 + 75 us at 128K tokens, 338 -> 99 + 118 at 64K and 50 %, 66 -> 48 + 13 at 32K).
//  1. Rows whose two largest block maxima the screen could not tell apart (ambmask) are settled
//     first: both blocks are re-evaluated with double-precision FMAs on the exact bf16 inputs,
//     which fixes the row's M* and which block(s) earn the HRM flag from that row (Eq. 12).
//  2. The candidates are ordered by (HRM flag descending, float32 score descending, block id
//     ascending).  Up to 128 of them: every key counts the keys above it, several threads a key.  More: they are dealt
//     into 33 buckets between 32 of 64 sorted sample keys, and every key counts the keys above it within its bucket; with a
//     small budget only the buckets of the order's head (the kept prefix plus a margin for step 3) are.
//  3. Two sorted neighbours with the same flag whose scores differ by less than tau_score
//     (relative) are a "near tie"; a maximal chain of near ties that starts inside the kept
//     prefix (or straddles its end) is left to be recounted in double precision (kap_recount.cuh): its entries go to the
//     list's row of scores, which is not needed any more.
// Everything outside such chains is ordered as exact arithmetic would order it provided the
// screen's error stays below tau_score / 2, which the tests check.  Query blocks the screen
// marked "hard", or with more chained entries than fit their row, go to the double-precision kernel.
#include <math.h>

#include "common.cuh"
#include "kap_recount.cuh"

namespace cosa {
namespace {

constexpr int kThreads = 128;
constexpr int kMaxRows = 64;   // sampled rows of one (possibly two-tile) query block
constexpr int kHeadCap = 256;     // entries of the order's head that are sorted on their own
constexpr int kAllPairs = 128;    // keys up to which every key is compared with every other
constexpr int kSamples = 64;      // sample keys, of which every second splits: 33 buckets
constexpr int kSplit = 32;
constexpr int kPerThread = 8;     // keys a thread keeps the place of
constexpr int kPad = kHeadDim + 4;   // row pitch in floats
constexpr int kTieMargin = 32;    // ... of which this many lie beyond the kept prefix

// Block maxima in double precision, straight from the bf16 keys; Qs holds the query block's sampled rows as floats, kPad apart.
// out[set][r] = max over the visible sampled keys c of block_of(set, r) of (Q~[r] . K~[c]) * scale, -inf when row r sees
// nothing of the block; entries whose block is negative are left alone.  A warp takes one row against one block: four
// lanes a key, eight keys at a time; (q0 + q1) + (q2 + q3) is the same in every lane.  All threads of the CTA call it.
template <typename BlockOf>
__device__ void f64_block_maxima(const KapParams& p, const float* Qs, int b, int g, int row0, int rows, int R, int n_sets,
                                 BlockOf block_of, double (*out)[kMaxRows], int tid) {
  const int lane = tid & 31, quarter = lane & 3;
  for (int item = tid >> 5; item < n_sets * rows; item += kThreads / 32) {
    const int set = item / rows, r = item % rows;
    const int j = block_of(set, r);
    if (j < 0) continue;                           // (the whole warp)
    double best = -INFINITY;
#pragma unroll 1
    for (int c0 = 0; c0 < R; c0 += 8) {
      const int kc = j * R + c0 + (lane >> 2);     // sampled key index
      const uint4* key = reinterpret_cast<const uint4*>(p.k + kv_off(p.pg, p.ks, b, p.hkv, g, kc * p.stride));
      double acc = 0.0;
#pragma unroll 2
      for (int u = 0; u < 4; ++u) {
        const uint4 w = key[u * 4 + quarter];
        const unsigned kw[4] = {w.x, w.y, w.z, w.w};
        const float* q = Qs + r * kPad + (u * 4 + quarter) * 8;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc = fma((double)q[2 * e], bf16_lo(kw[e]), acc);
          acc = fma((double)q[2 * e + 1], bf16_hi(kw[e]), acc);
        }
      }
      acc += __shfl_xor_sync(0xffffffffu, acc, 1);
      acc += __shfl_xor_sync(0xffffffffu, acc, 2);
      if (!p.causal || kc <= row0 + r) best = fmax(best, acc * p.scale);
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
    if (lane == 0) out[set][r] = best;
  }
  __syncthreads();
}

struct SortShared {
  unsigned long long samp[kSamples];
  unsigned split[kSplit], split_id[kSplit];             // upper (flag and score) and lower words of the splitters, descending: one bank each
  int start[kSplit + 2], cursor[kSplit + 1];            // by bucket: first position; keys so far
  int head_len;
};

// The bucket of a key: how many of the (descending) splitters lie above it.  The upper words decide, unless splitters share
// theirs (alike): many keys have one score then, as blocks whose exponentials all underflow to 0, and are parted by id.  In one
// bucket they would be compared all with all (Stage 1 of 2048 blocks of 4 heads, stride 16, Top-p, nine scores in ten 0: 2,311 us;
// parted 810, with the sorting network of before 1,088).
__device__ __forceinline__ int bucket_of(const SortShared* sh, unsigned long long key, bool alike) {
  const unsigned hi = (unsigned)(key >> 32);
  int b = 0;
#pragma unroll
  for (int step = kSplit / 2; step > 0; step >>= 1)
    if (sh->split[b + step - 1] > hi) b += step;
  b += sh->split[b] > hi ? 1 : 0;
  if (alike)
    while (b < kSplit && sh->split[b] == hi && sh->split_id[b] > (unsigned)key) ++b;
  return b;
}

// Sorts the distinct keys a[0 .. n) descending, at least the first `want` of them.  If the sorted head is shorter than n and
// fits kHeadCap it goes to head[] and a stays as it is; otherwise everything is sorted, in place.  Returns the length of the
// sorted part and sets *out to it.  tmp: n keys; bucket: n bytes.  one_bucket: as if no splitter were of any use (for
// tests).  All threads of the CTA call it.
// What counts is latency and shared-memory traffic: ten lists are in work on an SM (six when this was measured), each a chain of short steps between
// barriers.  A bitonic network (21 to 55 dependent rounds, one to eight warps) took 6.4 k cycles for 61 keys and 21 k for
// 512, a selection by pivots followed by a rank sort of the head 10.4 k for 1024; this takes 1.2, 7.8 and 6.6 k (Stage 1
// at 128K tokens 1540 -> 1425 us, at 64K and 50 % 724 -> 645, at 32K 207 -> 177, 61 blocks 85.5 -> 69.7).
__device__ int sort_head_desc(unsigned long long* a, int n, int want, unsigned long long* head, unsigned long long* tmp,
                              unsigned char* bucket, SortShared* sh, bool one_bucket, int tid, unsigned long long** out) {
  *out = a;
  if (n <= kAllPairs && !one_bucket) {
    int shift = 5;                                 // 2^shift threads per key (one for 65 to 128 keys)
    while ((n << shift) > kThreads) --shift;
    const int k = tid >> shift, part = tid & ((1 << shift) - 1);
    const unsigned long long key = k < n ? a[k] : 0ULL;
    int rank = 0;
#pragma unroll 4
    for (int u = part; u < n; u += 1 << shift) rank += (a[u] > key) ? 1 : 0;
    for (int o = (1 << shift) >> 1; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    __syncthreads();
    if (part == 0 && k < n) a[rank] = key;
    __syncthreads();
    return n;
  }
  // 64 samples, one from each stretch of n / 64 keys, ranked by two threads each
  if (tid < kSamples) {
    const int lo = (int)((long long)tid * n / kSamples), len = max(1, n / kSamples);
    sh->samp[tid] = a[lo + (tid * 5) % len];
  }
  if (tid <= kSplit) sh->cursor[tid] = 0;
  __syncthreads();
  if (one_bucket) {
    if (tid < kSplit) sh->split[tid] = ~0u;
  } else {
    static_assert(kThreads == 2 * kSamples, "two threads per sample");
    const unsigned long long mine = sh->samp[tid >> 1];
    int rank = 0;
#pragma unroll 8
    for (int u = 0; u < kSamples / 2; ++u) rank += (sh->samp[u * 2 + (tid & 1)] > mine) ? 1 : 0;
    rank += __shfl_xor_sync(0xffffffffu, rank, 1);
    if ((tid & 1) == 0 && (rank & 1)) { sh->split[rank >> 1] = (unsigned)(mine >> 32); sh->split_id[rank >> 1] = (unsigned)mine; }
  }
  __syncthreads();
  const int lane = tid & 31;
  const bool alike = !one_bucket && __any_sync(0xffffffffu, lane < kSplit - 1 && sh->split[lane] == sh->split[min(lane + 1, kSplit - 1)]);
  // every key to its bucket's count; a thread keeps bucket and place of its first eight keys (all there are up to 1024)
  unsigned place[kPerThread];
#pragma unroll
  for (int q = 0; q < kPerThread; ++q) {
    const int t = tid + q * kThreads;
    if (t < n) {
      const int b = bucket_of(sh, a[t], alike);
      place[q] = ((unsigned)b << 16) | (unsigned)atomicAdd(&sh->cursor[b], 1);
    }
  }
  if (n > kPerThread * kThreads) __syncthreads();     // (those come first in their buckets)
  for (int t = tid + kPerThread * kThreads; t < n; t += kThreads) atomicAdd(&sh->cursor[bucket_of(sh, a[t], alike)], 1);
  const int first_n = min(n, kPerThread * kThreads);
  __syncthreads();
  if (tid < 32) {                                  // where every bucket begins, and how many buckets the head takes
    const int c = sh->cursor[tid];
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (tid >= o) incl += v;
    }
    sh->start[tid] = incl - c;
    const int len = __reduce_min_sync(0xffffffffu, incl >= want ? incl : n);   // shortest run of whole buckets that holds `want` keys
    if (tid == 31) { sh->start[kSplit] = incl; sh->start[kSplit + 1] = n; }
    if (tid == 0) sh->head_len = len <= kHeadCap ? len : n;
  }
  __syncthreads();
  const int len = sh->head_len;
  // (bucket b is sorted iff it begins before `len`)
#pragma unroll
  for (int q = 0; q < kPerThread; ++q) {
    const int t = tid + q * kThreads;
    if (t < n) {
      const int b = (int)(place[q] >> 16), at = sh->start[b] + (int)(place[q] & 0xffffu);
      if (sh->start[b] < len) {
        tmp[at] = a[t];
        bucket[at] = (unsigned char)b;
      }
    }
  }
  if (n > first_n) {
    // more than 1024 keys: the rest finds its places again, from the ends of the buckets down (uniform over the CTA)
    for (int t = tid + first_n; t < n; t += kThreads) {
      const unsigned long long key = a[t];
      const int b = bucket_of(sh, key, alike);
      const int at = sh->start[b] + atomicSub(&sh->cursor[b], 1) - 1;
      if (sh->start[b] < len) {
        tmp[at] = key;
        bucket[at] = (unsigned char)b;
      }
    }
  }
  __syncthreads();
  unsigned long long* dst = len < n ? head : a;
  for (int t = tid; t < len; t += kThreads) {
    const unsigned long long key = tmp[t];
    const int b = bucket[t], first = sh->start[b], end = sh->start[b + 1];
    int rank = first;
    for (int u = first; u < end; ++u) rank += (tmp[u] > key) ? 1 : 0;
    dst[rank] = key;
  }
  __syncthreads();
  *out = dst;
  return len;
}

__global__ void __launch_bounds__(kThreads, 10) kap_sort_kernel(KapParams p, KapScreenParams sp, float tau_score, int sort_cap,
                                                            int tie_bytes, const int32_t* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(smem_raw);  // [sort_cap]
  unsigned char* tie = reinterpret_cast<unsigned char*>(keys + sort_cap);        // [tie_bytes]
  float* Qs = reinterpret_cast<float*>(tie + tie_bytes);                         // [R * tiles][kPad], filled on demand; the sort's
  unsigned long long* tmp = reinterpret_cast<unsigned long long*>(Qs);           // [sort_cap] scratch keys take the same place
  __shared__ double Mstar[kMaxRows];
  __shared__ double Mset[2][kMaxRows];
  __shared__ int j1[kMaxRows], j2[kMaxRows];
  __shared__ int n_tied, tail_end;
  __shared__ SortShared sort_sh;

  chain_begin();
  const int R = p.rows;                       // sampled rows per 128-row tile
  const int T = p.qtiles;                     // row tiles that share this ranking
  const int RT = R * T;
  const int big = p.nqb / T - 1 - (int)blockIdx.x;
  const int i_lo = big * T, i = i_lo + T - 1; // first and last row tile of the query block
  const int h = blockIdx.y, b = blockIdx.z;
  const int g = h / (p.hq / p.hkv);
  const int nqb_b = item_blocks(p.pg, b, p.nqb);   // the item's own length in blocks
  const int J = p.causal ? i + 1 : nqb_b;     // candidates: key blocks some row of the block may see
  const int tid = threadIdx.x;
  const size_t row_lo = (size_t)(b * p.hq + h) * p.nqb + i_lo;
  const size_t row = row_lo + (T - 1);
  // a screen kernel that gave up has left the scratch half written: nothing of it may be used for addressing
  const int poisoned = *reinterpret_cast<const volatile int32_t*>(status);   // (tested together with `hard` below)
  if (i >= nqb_b) {                           // padding past the item's length: empty lists
    if (poisoned != 0) return;
    for (int tile = 0; tile < T; ++tile) {
      for (int t = tid; t < p.order_stride; t += kThreads) p.order[(row_lo + tile) * p.order_stride + t] = -1;
      if (tid == 0) p.count[row_lo + tile] = 0;
    }
    return;
  }
  unsigned hard = 0u;                         // (tested only after the scores have been requested: one round trip, not two)
  float qk2 = 0.f;                            // largest product of squared norms of the block's sampled query rows and of its keys
  unsigned long long amb = 0ULL;              // bit r: sampled row r of the block was too close to call
  for (int t = 0; t < T; ++t) {
    hard |= sp.hard[row_lo + t];
    qk2 = fmaxf(qk2, sp.qk2max[row_lo + t]);
    amb |= (unsigned long long)sp.ambmask[row_lo + t] << (t * R);
  }
  int2 js = make_int2(0, 0);                  // (one round trip with the scores)
  if (tid < RT) js = reinterpret_cast<const int2*>(sp.jstar)[(size_t)(b * p.hq + h) * (p.n / p.stride) + (size_t)i_lo * R + tid];
  const __nv_bfloat16* qh = p.q + elem_off(p.qs, b, h, 0);

  // scores of the block = sum over its row tiles (the sum of Eq. 11 splits over the rows), flags = OR; a tile has
  // no score for key blocks wholly after it
  if (T == 1) {
    // eight scores per thread requested before any is used: the loads of a list are one round trip, not four
    const float* srow = sp.scores + row_lo * p.nqb;
    for (int j0 = 0; j0 < J; j0 += 8 * kThreads) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int j = j0 + u * kThreads + tid;
        v[u] = j < J ? srow[j] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int j = j0 + u * kThreads + tid;
        if (j < J) {
          const unsigned flag = (v[u] < 0.f) ? 0x80000000u : 0u;
          keys[j] = ((unsigned long long)(__float_as_uint(fabsf(v[u])) | flag) << 32) | (unsigned long long)(0xffffffffu - (unsigned)j);
        }
      }
    }
  } else {
    for (int j = tid; j < J; j += kThreads) {
      float sum = 0.f;
      unsigned flag = 0u;
      for (int t = 0; t < T; ++t) {
        if (p.causal && j > i_lo + t) continue;
        const float v = sp.scores[(row_lo + t) * p.nqb + j];
        sum += fabsf(v);
        flag |= (v < 0.f) ? 0x80000000u : 0u;
      }
      keys[j] = ((unsigned long long)(__float_as_uint(sum) | flag) << 32) | (unsigned long long)(0xffffffffu - (unsigned)j);
    }
  }
  if (poisoned != 0) return;
  // near ties: never closer than twice what the screen may be off by on rows of this magnitude
  tau_score = fmaxf(tau_score, 2.f * screen_error_bound(qk2, sp.scale));
  if (hard) {  // left to the double-precision kernel
    if (tid == 0) sp.entries[atomicAdd(sp.todo, 1)] = (int)row_lo;
    return;
  }
  if (tid == 0) { n_tied = 0; tail_end = 0; }
  if (tid < RT) { j1[tid] = js.x; j2[tid] = js.y; }
  __syncthreads();

  if (amb) {
    // ---- 1. settle the rows the screen could not call: set 0 = every row's best block, set 1 = the runner-up of
    // the rows in question
    if (tid < RT) Mset[1][tid] = -INFINITY;
    for (int e = tid; e < RT * (kHeadDim / 8); e += kThreads) {
      const int r = e / (kHeadDim / 8), c8 = e % (kHeadDim / 8);
      const uint4 w = reinterpret_cast<const uint4*>(qh + ((size_t)(i_lo * R + r) * p.stride) * p.qs.t)[c8];
      const unsigned ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        Qs[r * kPad + c8 * 8 + 2 * u] = __uint_as_float(ws[u] << 16);
        Qs[r * kPad + c8 * 8 + 2 * u + 1] = __uint_as_float(ws[u] & 0xffff0000u);
      }
    }
    __syncthreads();
    f64_block_maxima(p, Qs, b, g, i_lo * R, RT, R, 2,
                     [&](int set, int r) { return set == 0 ? j1[r] : (((amb >> r) & 1ULL) ? j2[r] : -1); }, Mset, tid);
    double* Msecond = Mset[1];
    if (tid < RT) Mstar[tid] = Mset[0][tid];
    __syncthreads();
    if (tid == 0) {
      for (int r = 0; r < RT; ++r) {
        if (!((amb >> r) & 1ULL)) continue;
        for (int which = 0; which < 2; ++which) {       // the HRM flag of both of the row's contenders
          const int j = which ? j2[r] : j1[r];
          bool flag = false;
          for (int q = 0; q < RT && !flag; ++q) {
            if ((amb >> q) & 1ULL) {
              const double best = fmax(Mstar[q], Msecond[q]);
              flag = (j == j1[q] && Mstar[q] == best) || (j == j2[q] && Msecond[q] == best);
            } else {
              flag = (j == j1[q]);
            }
          }
          keys[j] = (keys[j] & 0x7fffffffffffffffULL) | (flag ? 0x8000000000000000ULL : 0ULL);
        }
      }
    }
    __syncthreads();
  }
  if (p.dbg_scores || p.dbg_flags) {
    for (int j = tid; j < J; j += kThreads) {
      const unsigned hi = (unsigned)(keys[j] >> 32);
      if (p.dbg_scores) p.dbg_scores[row * p.nqb + j] = __uint_as_float(hi & 0x7fffffffu);
      if (p.dbg_flags) p.dbg_flags[row * p.nqb + j] = (unsigned char)(hi >> 31);
    }
    __syncthreads();
  }

  // ---- 2. order, descending in (flag, float32 score, -id).  With a small budget only the head of the order is
  // needed: the kept prefix plus a margin in which a chain of near ties that straddles its end can be followed.  A chain
  // that reaches the end of the sorted head (or Top-p, which needs the whole order) makes the rest follow.
  int K = budget_count_fx(p.budget_fx, J);
  __shared__ unsigned long long head[kHeadCap];
  __shared__ int need_full;
  const int want = p.sort_mode == 2 || p.top_p > 0.0 ? J : min(J, K + kTieMargin);
  unsigned long long* srt;          // the sorted order: srt[0 .. L)
  int L = sort_head_desc(keys, J, want, head, tmp, tie, &sort_sh, p.sort_mode == 1, tid, &srt);
  if (p.top_p > 0.0) {
      // Top-p retention: the shortest prefix of the order whose scores reach top_p of the total.  Every thread
      // owns a run of consecutive sorted entries; sums are double precision in a fixed order (deterministic).
      __shared__ double warp_sum[kThreads / 32];
      __shared__ int k_topp;
      const int E = (J + kThreads - 1) / kThreads;
      const int lane = tid & 31, wid = tid >> 5;
      double loc = 0.0;
      for (int q = 0; q < E; ++q) {
        const int t = tid * E + q;
        if (t < J) loc += (double)__uint_as_float((unsigned)(keys[t] >> 32) & 0x7fffffffu);
      }
      double incl = loc;
      for (int o = 1; o < 32; o <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      if (lane == 31) warp_sum[wid] = incl;
      if (tid == 0) k_topp = J;
      __syncthreads();
      double before = 0.0, total = 0.0;
      for (int w = 0; w < kThreads / 32; ++w) {
        if (w < wid) before += warp_sum[w];
        total += warp_sum[w];
      }
      const double thr = p.top_p * total;
      double run = before + (incl - loc);
      for (int q = 0; q < E; ++q) {
        const int t = tid * E + q;
        if (t >= J) break;
        run += (double)__uint_as_float((unsigned)(keys[t] >> 32) & 0x7fffffffu);
        if (run >= thr) { atomicMin(&k_topp, t + 1); break; }
      }
      __syncthreads();
      K = min(K, k_topp);
  }

  // ---- 3. near ties between sorted neighbours
  auto near_tie = [&](int t) {      // t + 1 < L
    const unsigned ha = (unsigned)(srt[t] >> 32), hb = (unsigned)(srt[t + 1] >> 32);
    if ((ha >> 31) != (hb >> 31)) return false;
    const float sa = __uint_as_float(ha & 0x7fffffffu), sb = __uint_as_float(hb & 0x7fffffffu);
    return sa - sb <= tau_score * sa;
  };
  // (none that begins inside the kept prefix: the usual case, and nothing more to do)
  bool any = false;
  for (int t = tid; t < K && t + 1 < L; t += kThreads) any = any || near_tie(t);
  if (__syncthreads_or(any)) {
    for (;;) {
      for (int t = tid; t < L; t += kThreads) tie[t] = t + 1 < L && near_tie(t) ? 1 : 0;
      __syncthreads();
      if (tid == 0) {  // a chain that straddles the end of the kept prefix reaches past it
        int e = K;
        while (e < L && tie[e - 1]) ++e;
        tail_end = e;
        need_full = (e == L && L < J) ? 1 : 0;   // the chain may go on beyond the sorted head
      }
      __syncthreads();
      if (!need_full) break;
      L = sort_head_desc(keys, J, J, head, tmp, tie, &sort_sh, p.sort_mode == 1, tid, &srt);
    }
    // entries: position, "tied with the next", id
    int* row_words = reinterpret_cast<int*>(sp.scores + row_lo * p.nqb);
    const int fit = max_chained(p.nqb * T, kRecountMax);
    for (int t = tid; t < tail_end; t += kThreads) {
      if ((t > 0 && tie[t - 1]) || tie[t]) {
        const int slot = atomicAdd(&n_tied, 1);
        if (slot < fit) {
          row_words[2 + slot] = chained_entry(t, tie[t], (int)(0xffffffffu - (unsigned)(srt[t] & 0xffffffffu)));
        }
      }
    }
    __syncthreads();
    const int nt = n_tied;
    if (nt > fit) {   // pathological: too many near ties
      if (tid == 0) sp.entries[atomicAdd(sp.todo, 1)] = (int)row_lo;
      return;
    }
    if (tid == 0 && nt > 0) {
      row_words[0] = nt; row_words[1] = K;
      sp.entries[p.batch * p.hq * p.nqb - 1 - atomicAdd(sp.todo + 1, 1)] = (int)row_lo;
    }
  }
  // the last row tile of the block takes the kept entries as they are; an earlier tile leaves out the key blocks that
  // lie wholly after it (with two tiles: the one block i), keeping the order
  __shared__ int pos_after;
  if (tid == 0) pos_after = K;
  __syncthreads();
  if (T == 2 && p.causal) {
    for (int t = tid; t < K; t += kThreads)
      if ((int)(0xffffffffu - (unsigned)(srt[t] & 0xffffffffu)) == i) pos_after = t;
    __syncthreads();
  }
  for (int tile = 0; tile < T; ++tile) {
    const bool drop = tile < T - 1 && pos_after < K;      // this tile leaves one entry out
    const int kept = K - (drop ? 1 : 0);
    int32_t* dst = p.order + (row_lo + tile) * p.order_stride;
    for (int t = tid; t < p.order_stride; t += kThreads) {
      const int src = (drop && t >= pos_after) ? t + 1 : t;
      dst[t] = (t < kept) ? (int32_t)(0xffffffffu - (unsigned)(srt[src] & 0xffffffffu)) : -1;
    }
    if (tid == 0) p.count[row_lo + tile] = kept;
  }
}

}  // namespace

cudaError_t launch_kap_sort(const KapParams& p, const KapScreenParams& sp, float tau_score, cudaStream_t st) {
  if (p.rows * p.qtiles > kMaxRows || p.nqb % p.qtiles != 0 || p.qtiles < 1 || p.qtiles > 2) return cudaErrorInvalidValue;
  const int cap = (p.nqb + 1) & ~1;            // keys, 16-byte pieces
  const int tie_bytes = (cap + 15) / 16 * 16;
  const size_t q_bytes = (size_t)p.rows * p.qtiles * kPad * 4, tmp_bytes = (size_t)cap * 8;
  const size_t smem = (size_t)cap * 8 + tie_bytes + (q_bytes > tmp_bytes ? q_bytes : tmp_bytes);
  static SmemLimit limit;
  cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(kap_sort_kernel), &limit, smem);
  if (e != cudaSuccess) return e;
  dim3 grid(p.nqb / p.qtiles, p.hq, p.batch);
  const int32_t* status = device_status_word();
  if (!status) return cudaErrorInvalidSymbol;
  return launch_chained(kap_sort_kernel, grid, kThreads, smem, st, p, sp, tau_score, cap, tie_bytes, status);
}

}  // namespace cosa
