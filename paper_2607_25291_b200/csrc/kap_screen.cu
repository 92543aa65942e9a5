// KAP fast path, stage A: the proxy scores on the sm_100a tensor cores (Sec. 4.2, Eqs. 8-12;
// Algorithm A steps 2-4).
//
// One CTA owns 256 sampled query rows = the R sampled rows of each of the G query heads of one
// KV head for 256/(G*R) consecutive query blocks, so that every sampled-key tile fetched once
// serves all of them: two row tiles of 128, because with a single one the kernel ran at the
// speed L2 could deliver key tiles, not at the speed of the tensor pipe.  The sampled logits of
// 128 rows x 128 sampled keys (= 128/R key blocks) are one tcgen05 MMA tile with a TMEM
// accumulator; strided TMA boxes gather every s-th row of Q and K directly (the down-sampled
// matrices are never materialised).
//
// The row maximum M*[r] must be known before Pbar[r,j] = exp(M[r,j] - M*[r]) can be summed, and
// the per-row block maxima of 256 rows do not fit on chip at long context.  The contraction is
// still done once: while the key tiles stream by, every epilogue thread takes its row's block
// maxima M[r,j] (tracking the three largest and the blocks holding the two largest) and parks
// them in a scratch area of global memory that the CTA owns while it runs; there are only as
// many such areas as CTAs can be resident, so they mostly stay in L2.  After the last tile, with
// M* known, the block scores and HRM flags are formed from the parked maxima, one thread per
// (row group, key block).
// Calls of at most four key tiles (512 sampled keys) park nothing, nor do those of at most eight whose lists are made here and whose
// blocks have 16 sampled rows or more: a thread keeps its block maxima in registers and, when
// every product is done, lays them into the key stages, from where the scores are formed; the norms of the sampled keys are
// taken from the stages as well, which saves the norms kernel's launch.
// A CTA holds every score of its lists, and up to 256 candidates it sorts them itself, a warp a list in registers (list_sort.cuh): no sort
// kernel (a wave of small CTAs each, chains of short steps between barriers), and no scores cross a launch, only the lists (a byte an
// entry).  Against the sort kernel Stage 1 took 135 us instead of 160 at 32K, 58 instead of 102 for 55 blocks at stride 4, 43 instead of 70
// for 2 x 61 blocks of 32 heads.
// What bounds the tiles of long calls: the tensor pipe, which takes 1,139 cycles of an SM a key tile for two products; with both operands
// in shared memory and 128 columns a product takes 570 or more, not 512.  (Issued under lane == 0, not elect.sync, a tile took 1,518.)
// A CTA at 32K (16.5 tiles): 41,400 cycles, of them 6,600 to the first logits, 19,000 for tiles, 1,700 for M* and thresholds, 5,700 for
// scores, 7,500 for lists; at 128K (64.5 tiles) 97,000, scores 16,000.  Short calls are a chain of latencies: launch, first loads, a wave
// or two of CTAs.  What a CTA needs once has two warps of its own, which work while products run (by the epilogue warps first: 129 us at
// 32K instead of 124, 14.1 for 31 blocks of 32 heads instead of 12.9).
// Float32 results are a SCREEN: the sort stage recomputes in double precision whatever a
// rounding error could reorder.  For that it is told, per sampled row, the two blocks with the
// largest block maxima and whether they are closer than tau_row (the row's HRM flag and M* are
// then settled in double precision); three such blocks on one row send the whole query block to
// the double-precision kernel.
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "kap_recount.cuh"
#include "list_sort.cuh"
#include "ptx_sm100.cuh"
#include "tile_maps.cuh"

namespace cosa {
namespace {

using namespace ptx;

constexpr int kStages = 4;
constexpr int kTileBytes = 128 * kHeadDim * 2;
constexpr int kHalfBytes = kTileBytes / 2;
constexpr int kRowTiles = 2;          // 128-row tiles of sampled queries per CTA
constexpr int kRows = 128 * kRowTiles;
constexpr int kParts = 2;             // column parts of a tile: one epilogue warp per row tile, part and sub-partition
constexpr int kPartCols = 128 / kParts;
constexpr int kEpiThreads = 128 * kRowTiles * kParts;
constexpr int kAuxThreads = 64;       // two warps for what a CTA needs once: scratch area, norms
constexpr int kThreads = 64 + kEpiThreads + kAuxThreads;    // producer warp, MMA warp, epilogue warps, aux warps
constexpr int kSteps = 2;             // key tiles whose logits are in tensor memory at once
constexpr int kTmemCols = 128 * kRowTiles * kSteps;
// 20 warps, five a scheduler: a thread has 96 registers.  The forms spill up to 24 bytes (loads: up to 32, of the long form with lists and 32
// sampled rows a block 64)
constexpr int kCtasPerSm = 1;
static_assert(kTmemCols == 512 && kPartCols == 64, "TMEM budget and two 32-column loads per thread and tile");

struct __align__(8) ScreenCtl {
  unsigned long long a_full, k_full[kStages];
  unsigned long long k_empty[kStages];  // the tile's MMAs finished: stage free and logits ready
  unsigned long long s_empty[kSteps];
  unsigned long long slot_bar;          // the CTA has its scratch area
  unsigned long long norm_bar;          // norms are there
  unsigned long long parked_bar;        // every maximum of the CTA is parked
  unsigned long long m_full[kStages], m_empty[kStages];   // parked maxima fetched back into a key stage / read by all
  uint32_t tmem_base;
  volatile int abort_flag;
  volatile int t_issued, t_done, c_fetched, c_done;   // key tiles requested / multiplied, chunks of parked maxima requested / read
  int slot;                             // scratch area held by this CTA, -1 = none
  bool poisoned;                        // some CTA has reported a timeout: this one does nothing
  float xt[kParts][3][kRows];           // exchange between the column parts: top-3 block maxima
  int xj[kParts][2][kRows];             // ... and the blocks holding the two largest
  float mstar[kRows];                   // M*[r] of every row
  float q2[kParts][kRows];              // squared norm of every row (by two threads, half a row each, or whole in the first)
  float k2w[kAuxThreads / 32];          // largest squared key norm each aux warp saw
  unsigned long long n_read[kStages];   // (kMedium) both aux warps have the norms of the stage's keys
  int j12[2][kRows];                    // (lists) blocks holding every row's largest and second largest block maximum
  uint32_t amb[kRows / 8];              // (lists) by row group: rows whose two best blocks are too close to call
  float qk2[kRows / 8];                 // (lists) by row group: as qk2max
  bool hard[kRows / 8];                 // (lists) by row group: as `hard`
};
constexpr size_t kScreenSmem = 1024 + (size_t)kTileBytes * (kRowTiles + kStages) + sizeof(ScreenCtl);
static_assert(kScreenSmem <= 232448, "shared memory budget of one CTA");

__device__ __forceinline__ void screen_timeout(ScreenCtl* c, int32_t* status) {
  c->abort_flag = 1;
  atomicMin(status, (int32_t)COSA_ERR_DEVICE_TIMEOUT);
}

// Takes a scratch area if it is free; what its last holder did with it has happened then
__device__ __forceinline__ bool take_area(int32_t* taken) {
  int32_t was;
  asm volatile("atom.acquire.gpu.global.cas.b32 %0, [%1], 0, 1;" : "=r"(was) : "l"(taken) : "memory");
  return was == 0;
}

// (a whole warp) the largest squared norm of a sampled key row of the call
__device__ __forceinline__ float largest_key_norm(const KapScreenParams& p, int lane) {
  float k2 = 0.f;
  for (int t = lane; t < p.k2parts; t += 32) k2 = fmaxf(k2, p.k2part[t]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) k2 = fmaxf(k2, __shfl_xor_sync(0xffffffffu, k2, o));
  return k2;
}

constexpr int kMediumTiles = 8;           // key tiles of a call of the medium form
constexpr int kListCap = 64, kLongListCap = 256;   // candidates a list may have where this kernel makes the lists
constexpr bool rows_hold_lists() {
  for (int nqb = 1; nqb <= kLongListCap; ++nqb) {
    const int chained = max_chained(nqb, kRecountMax);
    if (list_words(nqb) > nqb || (chained >= 2 && 2 + chained + list_words(nqb) > nqb)) return false;   // (a chain has two entries at least)
  }
  return true;
}
static_assert(rows_hold_lists(), "a row of scores holds a list and the entries of its near ties");

// (a whole warp) the largest of row `qrow` x the sampled keys that the row sees of block j[0] and of block j[1], in double precision:
// the arithmetic of f64_block_maxima in kap_sort.cu, the row taken from global memory.  Bound by round
// trips to L2, with few warps to hide them, and by the conversions: the loads of both blocks and of 16 keys of each go out together, of
// kAhead quarters of their 256 bytes (one block, 8 keys and a quarter at a time, with every block the copy of another: Stage 1 of 31
// blocks of 32 heads 187 us instead of 138, of 200 blocks 2,097 instead of 1,940, of 8 blocks of 2 heads, whose rows all lie in one
// CTA, 108 instead of 67; there the sort kernel, impl = 3, takes 56)
template <int R, int kAhead>
__device__ __forceinline__ void f64_row_maxima(const KapParams& p, const __nv_bfloat16* qrow, int b, int g, const int (&j)[2], int r_glob,
                                               int lane, double (&best)[2]) {
  constexpr int kKeys = R < 16 ? 1 : 2;
  const int quarter = lane & 3;
  best[0] = best[1] = -INFINITY;
#pragma unroll 1
  for (int c0 = 0; c0 < R; c0 += 8 * kKeys) {
    const uint4* key[2][kKeys];
    double acc[2][kKeys];
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
      for (int c = 0; c < kKeys; ++c) {
        key[x][c] = reinterpret_cast<const uint4*>(p.k + kv_off(p.pg, p.ks, b, p.hkv, g, (j[x] * R + c0 + 8 * c + (lane >> 2)) * p.stride)) + quarter;
        acc[x][c] = 0.0;
      }
#pragma unroll kAhead
    for (int u = 0; u < 4; ++u) {
      const uint4 q = reinterpret_cast<const uint4*>(qrow)[u * 4 + quarter];
      const unsigned qw[4] = {q.x, q.y, q.z, q.w};
      uint4 w[2][kKeys];
#pragma unroll
      for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int c = 0; c < kKeys; ++c) w[x][c] = key[x][c][u * 4];
#pragma unroll
      for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int c = 0; c < kKeys; ++c) {
          const unsigned kw[4] = {w[x][c].x, w[x][c].y, w[x][c].z, w[x][c].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            acc[x][c] = fma(bf16_lo(qw[e]), bf16_lo(kw[e]), acc[x][c]);
            acc[x][c] = fma(bf16_hi(qw[e]), bf16_hi(kw[e]), acc[x][c]);
          }
        }
    }
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
      for (int c = 0; c < kKeys; ++c) {
        double z = acc[x][c];
        z += __shfl_xor_sync(0xffffffffu, z, 1);
        z += __shfl_xor_sync(0xffffffffu, z, 2);
        if (!p.causal || j[x] * R + c0 + 8 * c + (lane >> 2) <= r_glob) best[x] = fmax(best[x], z * p.scale);
      }
  }
#pragma unroll
  for (int x = 0; x < 2; ++x)
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) best[x] = fmax(best[x], __shfl_xor_sync(0xffffffffu, best[x], o));
}

// (a whole warp) the visit list of one (head, query block) of at most 32 * PER candidates: what kap_sort_kernel does for longer
// calls, step by step.  score[j]: the screened scores (sign: HRM flag); j1, j2: its rows' best and second best blocks; srt: room for
// the keys.  The list waits in its row of `scores`; what is left for the fix-up: near ties (entries in the same row) or the whole list.
// sp.hard says so, and without kFlags the worklist, too
template <int R, int PER, bool kFlags>
__device__ void make_list(const KapParams& p, const KapScreenParams& sp, float tau_score, int b, int g, int h, int i, int J, uint32_t amb,
                          bool hard, float qk2, const float* score, const int* j1, const int* j2, unsigned long long* srt, int lane) {
  const size_t row = (size_t)(b * p.hq + h) * p.nqb + i;
  auto leave = [&](ListState state) {
    if (lane != 0) return;
    sp.hard[row] = (uint8_t)state;
    if (kFlags) return;
    if (state == kListRedo) sp.entries[atomicAdd(sp.todo, 1)] = (int)row;
    else if (state == kListTies) sp.entries[p.batch * p.hq * p.nqb - 1 - atomicAdd(sp.todo + 1, 1)] = (int)row;
  };
  if (hard) {                               // three-way row ambiguity: left to the double-precision kernel
    leave(kListRedo);
    return;
  }
  unsigned long long key[PER];
#pragma unroll
  for (int x = 0; x < PER; ++x) {
    const int j = lane + 32 * x;
    const float v = j < J ? score[j] : 0.f;
    key[x] = j < J ? ((unsigned long long)(__float_as_uint(fabsf(v)) | (v < 0.f ? 0x80000000u : 0u)) << 32) | (0xffffffffu - (unsigned)j) : 0ULL;
  }
  if (amb) {
    // rows the screen could not call: which of their two blocks holds the maximum, and so which earn the HRM flag (lane r: row r)
    double m1 = -INFINITY, m2 = -INFINITY;
    const int a1 = lane < R ? j1[lane] : -1, a2 = lane < R ? j2[lane] : -1;
    const __nv_bfloat16* qh = p.q + elem_off(p.qs, b, h, 0);
#pragma unroll 1
    for (uint32_t left = amb; left; left &= left - 1) {
      const int r = __ffs(left) - 1;
      const __nv_bfloat16* qrow = qh + (long long)(i * R + r) * p.stride * p.qs.t;
      const int two[2] = {j1[r], j2[r]};
      double z[2];
      f64_row_maxima<R, kFlags ? 4 : 1>(p, qrow, b, g, two, i * R + r, lane, z);   // (the long form has no registers for more)
      if (lane == r) { m1 = z[0]; m2 = z[1]; }
    }
    const double best = fmax(m1, m2);
    const bool mine = lane < R && ((amb >> lane) & 1u);
#pragma unroll 1
    for (uint32_t left = amb; left; left &= left - 1) {
      const int r = __ffs(left) - 1;
#pragma unroll 1
      for (int which = 0; which < 2; ++which) {
        const int j = which ? j2[r] : j1[r];
        const bool flag = __any_sync(0xffffffffu, lane < R && (mine ? (j == a1 && m1 == best) || (j == a2 && m2 == best) : j == a1));
#pragma unroll
        for (int x = 0; x < PER; ++x)
          if (j == lane + 32 * x) key[x] = (key[x] & 0x7fffffffffffffffULL) | (flag ? 0x8000000000000000ULL : 0ULL);
      }
    }
  }
  if (p.dbg_scores || p.dbg_flags) {
#pragma unroll
    for (int x = 0; x < PER; ++x) {
      const int j = lane + 32 * x;
      const unsigned hi = (unsigned)(key[x] >> 32);
      if (j < J && p.dbg_scores) p.dbg_scores[row * p.nqb + j] = __uint_as_float(hi & 0x7fffffffu);
      if (j < J && p.dbg_flags) p.dbg_flags[row * p.nqb + j] = (unsigned char)(hi >> 31);
    }
  }
  if (PER == 2 && J <= 16) {                // (every key counts the keys above it: fewer steps than the sort of 64)
    int rank = 0;
#pragma unroll 4
    for (int u = 0; u < J; ++u) rank += __shfl_sync(0xffffffffu, key[0], u) > key[0] ? 1 : 0;
    if (lane < J) srt[rank] = key[0];
  } else {
    sort_list<PER>(key, score, J, srt, lane);
  }
  __syncwarp();
  auto score_at = [&](int t) { return __uint_as_float((unsigned)(srt[t] >> 32) & 0x7fffffffu); };
  int K = budget_count_fx(p.budget_fx, J);
  if (p.top_p > 0.0) {
    // Top-p: the sums of kap_sort_kernel, where each of 128 threads has E consecutive entries; x: its warps
    constexpr int kWarps = PER < 4 ? PER : 4;
    const int E = (J + 127) / 128;
    double start[kWarps], total = 0.0;
#pragma unroll
    for (int x = 0; x < kWarps; ++x) {
      start[x] = 0.0;
      if (32 * x * E >= J) continue;
      const int t0 = (32 * x + lane) * E;
      double loc = 0.0;
      for (int q = 0; q < E; ++q)
        if (t0 + q < J) loc += (double)score_at(t0 + q);
      double incl = loc;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      start[x] = total + (incl - loc);
      total += __shfl_sync(0xffffffffu, incl, 31);
    }
    const double thr = p.top_p * total;
    unsigned k_topp = (unsigned)J;
#pragma unroll
    for (int x = 0; x < kWarps; ++x) {
      const int t0 = (32 * x + lane) * E;
      double run = start[x];
      for (int q = 0; q < E && t0 + q < J; ++q) {
        run += (double)score_at(t0 + q);
        if (run >= thr) { k_topp = min(k_topp, (unsigned)(t0 + q + 1)); break; }
      }
    }
    K = min(K, (int)__reduce_min_sync(0xffffffffu, k_topp));
  }
  // near ties between sorted neighbours
  tau_score = fmaxf(tau_score, 2.f * screen_error_bound(qk2, sp.scale));
  uint32_t tie[PER];                        // bit l of tie[x]: entries t = 32 x + l and t + 1
  bool any = false;
#pragma unroll
  for (int x = 0; x < PER; ++x) {
    const int t = lane + 32 * x;
    bool near = false;
    if (t + 1 < J) {
      const unsigned ha = (unsigned)(srt[t] >> 32), hb = (unsigned)(srt[t + 1] >> 32);
      const float sa = __uint_as_float(ha & 0x7fffffffu), sb = __uint_as_float(hb & 0x7fffffffu);
      near = (ha >> 31) == (hb >> 31) && sa - sb <= tau_score * sa;
    }
    any = any || (near && t < K);
    tie[x] = __ballot_sync(0xffffffffu, near);
  }
  ListState state = kListMade;
  if (__any_sync(0xffffffffu, any)) {
    int e = K;                              // a chain that straddles the end of the kept prefix reaches past it
    bool more = true;
#pragma unroll
    for (int x = 0; x < PER; ++x) {
      while (more && e > 32 * x && e <= 32 * x + 32 && e < J) {
        more = (tie[x] >> ((e - 1) & 31)) & 1u;
        e += more ? 1 : 0;
      }
    }
    int nt = 0;
    uint32_t members[PER];
#pragma unroll
    for (int x = 0; x < PER; ++x) {
      const int n = e - 32 * x;             // entries of this word before e
      const uint32_t below = n >= 32 ? ~0u : (n <= 0 ? 0u : (1u << n) - 1u);
      members[x] = (tie[x] | (tie[x] << 1) | (x > 0 ? tie[x > 0 ? x - 1 : 0] >> 31 : 0u)) & below;
      nt += __popc(members[x]);
    }
    if (nt > max_chained(p.nqb, kRecountMax)) {
      leave(kListRedo);
      return;
    }
    int* words = reinterpret_cast<int*>(sp.scores + row * p.nqb);
    if (lane == 0) { words[0] = nt; words[1] = K; }
    int slot0 = 0;
#pragma unroll
    for (int x = 0; x < PER; ++x) {
      if ((members[x] >> lane) & 1u) {
        const int slot = slot0 + __popc(members[x] & ((1u << lane) - 1u)), t = lane + 32 * x;
        words[2 + slot] = chained_entry(t, (int)((tie[x] >> lane) & 1u), (int)(0xffffffffu - (unsigned)srt[t]));
      }
      slot0 += __popc(members[x]);
    }
    state = kListTies;
  }
  const int n_words = list_words(p.nqb);
  uint32_t* kept = reinterpret_cast<uint32_t*>(sp.scores + (row + 1) * p.nqb - n_words);
  for (int w = lane; w < n_words; w += 32) {
    uint32_t bytes = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int t = 4 * w + e;
      bytes |= (t < K ? 0xffu - ((unsigned)srt[t] & 0xffu) : (t == p.nqb ? (unsigned)K - 1u : 0u)) << (8 * e);
    }
    kept[w] = bytes;
  }
  leave(state);
}

// kStrict: the call's budget for waits is short; waits are polled and answer per warp (see mbar_poll).  kForm: see above
template <int R, bool kStrict, int kForm>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
kap_screen_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                  KapScreenParams p, KapParams kp, float tau_score, int32_t* status) {
  constexpr bool kLongLists = kForm == kScreenLongLists, kOnChip = kForm != kScreenLong && !kLongLists, kMedium = kForm == kScreenMediumLists;
  constexpr bool kLists = kForm == kScreenShortLists || kMedium || kLongLists;
  constexpr int kMaxTiles = kMedium ? kMediumTiles : kStages;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (base - raw);
  const uint32_t a_sm = base;
  const uint32_t k_sm = base + kRowTiles * kTileBytes;
  ScreenCtl* ctl = reinterpret_cast<ScreenCtl*>(smem + (size_t)kTileBytes * (kRowTiles + kStages));
  // what needs nothing of the kernel before
  if (threadIdx.x == 0) {
    prefetch_tensormap(&q_map); prefetch_tensormap(&k_map);
    mbar_init(smem_u32(&ctl->a_full), 1);
    for (int s = 0; s < kStages; ++s) { mbar_init(smem_u32(&ctl->k_full[s]), 1); mbar_init(smem_u32(&ctl->k_empty[s]), 1); }
    for (int s = 0; s < kSteps; ++s) mbar_init(smem_u32(&ctl->s_empty[s]), kEpiThreads);
    mbar_init(smem_u32(&ctl->norm_bar), kAuxThreads / 32);
    mbar_init(smem_u32(&ctl->slot_bar), 1); mbar_init(smem_u32(&ctl->parked_bar), 1);
    if (!kOnChip) for (int s = 0; s < kStages; ++s) { mbar_init(smem_u32(&ctl->m_full[s]), 1); mbar_init(smem_u32(&ctl->m_empty[s]), kEpiThreads); }
    if (kMedium) for (int s = 0; s < kStages; ++s) mbar_init(smem_u32(&ctl->n_read[s]), kAuxThreads / 32);
    ctl->abort_flag = 0;
    ctl->t_issued = 0; ctl->t_done = 0; ctl->c_fetched = 0; ctl->c_done = 0;
    mbar_fence_init();
    fence_proxy_async_smem();
  }
  __syncwarp();
  chain_wait();

  constexpr int BPT = 128 / R;                  // key blocks per key tile
  constexpr int kGroups = kRows / R;            // row groups (one query head of one query block each) per CTA
  const int lg = p.group_shift, G = 1 << lg;    // query heads of the group (a power of two: see kap_screen_supported)
  const int QB = kGroups >> lg;                 // query blocks per CTA
  const int n_iq = p.n_iq;
  const int bg = (int)blockIdx.x / n_iq;
  const int b = bg / p.hkv;
  const int g = bg - b * p.hkv;
  const int iq = n_iq - 1 - ((int)blockIdx.x - bg * n_iq);   // longest first
  const int i0 = iq * QB;
  const int nqb_b = item_blocks(p.pg, b, p.nqb);      // the item's own length in blocks
  const int i_max = min(i0 + QB, nqb_b) - 1;
  const int ns = p.nqb * R;                     // sampled rows per head (tensor pitch)
  const int ns_b = nqb_b * R;                   // ... that the item really has
  const int n_keys = p.causal ? (i_max + 1) * R : ns_b;
  const int n_tiles = (n_keys + 127) / 128;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (uniform, which the compiler cannot know)

  if (!kLists && blockIdx.x == 0 && threadIdx.x == 0) { p.todo[0] = 0; p.todo[1] = 0; }   // the sort stage (a later launch) counts there
  if (kLists && threadIdx.x < kGroups) {          // query blocks that are padding: empty lists
    const int x = threadIdx.x, i = i0 + (x >> lg);
    if (i >= nqb_b && i < p.nqb) p.hard[(size_t)(b * p.hq + g * G + (x & (G - 1))) * p.nqb + i] = kListPadding;
  }
  if (i0 >= nqb_b) return;                        // all of this CTA's query blocks are padding
  // key tile t to its stage: by one thread, or, with pages, by a whole warp (the 128 sampled keys of a tile come from 128 / spp pages,
  // spp sampled rows each, or from one page; one lane per page looks its page up and issues its two boxes.  Sampled keys past the
  // sequence are masked later: any valid page will do for them)
  auto fetch_dense = [&](int t) {
    const int st = t % kStages;
    const uint32_t dst = k_sm + st * kTileBytes, bar = smem_u32(&ctl->k_full[st]);
    mbar_expect_tx(bar, kTileBytes);
    tma_load_tile(dst, &k_map, 0, t * 128, g, b, p.ko.row, p.ko.head, p.ko.outer, bar);
    tma_load_tile(dst + kHalfBytes, &k_map, 64, t * 128, g, b, p.ko.row, p.ko.head, p.ko.outer, bar);
  };
  auto fetch_pages = [&](int t) {
    const int st = t % kStages;
    const uint32_t dst = k_sm + st * kTileBytes, bar = smem_u32(&ctl->k_full[st]);
    if (elect_one()) mbar_expect_tx(bar, kTileBytes);
    __syncwarp();
    const int spp = min(128, p.pg.page_size / p.stride);
    if (lane < 128 / spp) {
      int tok = (t * 128 + lane * spp) * p.stride;
      if (tok >= nqb_b * kBlock) tok = 0;
      const KvCoord c = kv_coord(p.pg, b, g, tok);        // (a page's first sampled row is a multiple of the stride)
      tma_load_tile(dst + lane * spp * 128, &k_map, 0, c.row / p.stride, c.head, c.outer, p.ko.row, p.ko.head, p.ko.outer, bar);
      tma_load_tile(dst + kHalfBytes + lane * spp * 128, &k_map, 64, c.row / p.stride, c.head, c.outer, p.ko.row, p.ko.head, p.ko.outer, bar);
    }
    __syncwarp();
  };
  const int n_first = min(n_tiles, 1);            // (a tile takes its thread some 500 cycles)
  if (warp == 0) {
    // The first tiles at once; tensor memory, the status word and a scratch area come meanwhile (one after the other a CTA spent
    // 4,300 cycles before its first request: Stage 1 at 32K 169 -> 167 us, of 4K tokens of 4 heads 17.4 -> 16.6).
    // A tiles: strided boxes of R sampled rows of q_box_heads query heads of the group (all of them, if the layout has rows
    // inside heads) per query block, a box pair per lane (one lane issuing 32 boxes in turn: 2 us)
    if (lane == 0) mbar_expect_tx(smem_u32(&ctl->a_full), kRowTiles * kTileBytes);
    __syncwarp();
    static_assert(kGroups <= 32, "a lane per box pair");
    const int a_grp = lane * p.q_box_heads;
    if (a_grp < kGroups) {
      const int i = i0 + (a_grp >> lg), h = g * G + (a_grp & (G - 1));
      const uint32_t dst = a_sm + (a_grp * R / 128) * kTileBytes + (a_grp * R % 128) * 128;   // (rows past the head's last are zero-filled)
      tma_load_tile(dst, &q_map, 0, i * R, h, b, p.qo.row, p.qo.head, p.qo.outer, smem_u32(&ctl->a_full));
      tma_load_tile(dst + kHalfBytes, &q_map, 64, i * R, h, b, p.qo.row, p.qo.head, p.qo.outer, smem_u32(&ctl->a_full));
    }
    __syncwarp();
    if (n_first > 0) {
      if (p.pg.table) fetch_pages(0);
      else if (elect_one()) fetch_dense(0);
    }
  } else if (warp == 1) {
    tmem_alloc(smem_u32(&ctl->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  chain_next();                            // (tensor memory is allocated)
  const uint32_t tmem = ctl->tmem_base;
  volatile int* abort_flag = &ctl->abort_flag;
  const long long budget = p.wait_budget;
  auto wait = [&](uint32_t bar, uint32_t parity) {
    return kStrict ? mbar_poll(bar, parity, abort_flag, budget) : mbar_wait(bar, parity, abort_flag, budget);
  };
  auto wait_warp = [&](uint32_t bar, uint32_t parity) {
    return kStrict ? mbar_poll_warp(bar, parity, abort_flag, budget) : mbar_wait(bar, parity, abort_flag, budget);
  };

  // squared norm of the row of a tile at `row`, 128 bytes of it or all 256, the other half a half tile further on (the swizzle permutes
  // 16-byte chunks inside 128 bytes, which a sum of squares does not notice; the chunk order is rotated by the lane so that the rows
  // of a warp hit different banks)
  auto norm2 = [&](const unsigned char* row, auto chunks) {
    unsigned long long s0 = pack_f32x2(0.f, 0.f), s1 = s0;
#pragma unroll
    for (int c = 0; c < decltype(chunks)::value; ++c) {
      const uint4 wv = *reinterpret_cast<const uint4*>(row + (c >> 3) * kHalfBytes + (((c + lane) & 7) << 4));
      const unsigned ws4[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const unsigned long long two = pack_f32x2(__uint_as_float(ws4[u] << 16), __uint_as_float(ws4[u] & 0xffff0000u));
        if (u & 1) s1 = fma_f32x2(two, two, s1); else s0 = fma_f32x2(two, two, s0);
      }
    }
    float x, y;
    unpack_f32x2(add_f32x2(s0, s1), x, y);
    return x + y;
  };

  if (warp == 0) {
    int t_issued = n_first;
    if (!p.pg.table) {
      if (elect_one()) {
        for (int t = n_first; t < n_tiles; ++t) {
          const int st = t % kStages;
          if (!wait(smem_u32(&ctl->k_empty[st]), ((t / kStages) & 1) ^ 1) ||
              (kMedium && !wait(smem_u32(&ctl->n_read[st]), ((t / kStages) & 1) ^ 1))) {
            if (!*abort_flag) screen_timeout(ctl, status);
            break;
          }
          fetch_dense(t);
          t_issued = t + 1;
        }
        ctl->t_issued = t_issued;
      }
    } else {
      for (int t = n_first; t < n_tiles; ++t) {
        const int st = t % kStages;
        int ok = 1;
        if (lane == 0) {
          ok = wait(smem_u32(&ctl->k_empty[st]), ((t / kStages) & 1) ^ 1) ? 1 : 0;
          if (kMedium && ok) ok = wait(smem_u32(&ctl->n_read[st]), ((t / kStages) & 1) ^ 1) ? 1 : 0;
          if (!ok && !*abort_flag) screen_timeout(ctl, status);
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) break;
        fetch_pages(t);
        t_issued = t + 1;
      }
      if (lane == 0) ctl->t_issued = t_issued;
    }
    __syncwarp();
    if (!kOnChip && elect_one()) {
      // the parked maxima come back through the key stages, a chunk of tiles each, when every one of them is parked
      int c_fetched = 0;
      bool alive = wait(smem_u32(&ctl->parked_bar), 0);
      if (alive) {
        const float* parked = p.maxima + (size_t)ctl->slot * ((size_t)((ns + 127) / 128) * (kRows * BPT));
        const uint64_t drop = l2_policy_evict_first();
        fence_proxy_async_all();   // the maxima were written with ordinary stores
        constexpr int kTileFloats = kRows * BPT, kTilesPerChunk = kTileBytes / (kTileFloats * 4);
        const int n_chunks = (n_tiles + kTilesPerChunk - 1) / kTilesPerChunk;
        for (int c = 0; c < n_chunks; ++c) {
          const int st = c % kStages;
          if (c >= kStages) alive = wait(smem_u32(&ctl->m_empty[st]), ((c - kStages) / kStages) & 1);
          if (!alive) break;
          const int tiles_here = min(kTilesPerChunk, n_tiles - c * kTilesPerChunk);
          const uint32_t bar = smem_u32(&ctl->m_full[st]);
          mbar_expect_tx(bar, tiles_here * kTileFloats * 4);
          bulk_load_hint(k_sm + st * kTileBytes, parked + (size_t)c * kTilesPerChunk * kTileFloats, tiles_here * kTileFloats * 4, bar, drop);
          c_fetched = c + 1;
        }
      }
      if (!alive && !*abort_flag) screen_timeout(ctl, status);
      ctl->c_fetched = c_fetched;
    }
  } else if (warp == 1) {
    if (elect_one()) {
      const uint32_t idesc = idesc_bf16(128, 128, 0, 0);
      bool alive = wait(smem_u32(&ctl->a_full), 0);
      if (!alive && !*abort_flag) screen_timeout(ctl, status);
      int t_done = 0;
      // (the barriers of the next tile are looked at between the products on this one's row tiles: asked behind them, the tensor
      // pipe would idle for as long as two waits take)
      bool k_here = false, s_here = false;
      for (int t = 0; t < n_tiles && alive; ++t) {
        const int st = t % kStages, sb = t % kSteps, st1 = (t + 1) % kStages, sb1 = (t + 1) % kSteps;
        alive = (k_here || wait(smem_u32(&ctl->k_full[st]), (t / kStages) & 1)) &&
                (s_here || wait(smem_u32(&ctl->s_empty[sb]), ((t / kSteps) & 1) ^ 1));
        if (!alive) { if (!*abort_flag) screen_timeout(ctl, status); break; }
        tc_fence_after();
        const uint64_t kdesc = smem_desc_sw128(k_sm + st * kTileBytes, 16, 1024);
#pragma unroll
        for (int rt = 0; rt < kRowTiles; ++rt) {
          mma_ss_x8<2, 4, 6, kHalfBytes / 16, kHalfBytes / 16 + 2, kHalfBytes / 16 + 4, kHalfBytes / 16 + 6>(
              tmem + (sb * kRowTiles + rt) * 128, smem_desc_sw128(a_sm + rt * kTileBytes, 16, 1024), kdesc, idesc);
          if (rt == 0) {
            k_here = mbar_test_wait(smem_u32(&ctl->k_full[st1]), ((t + 1) / kStages) & 1);
            s_here = mbar_test_wait(smem_u32(&ctl->s_empty[sb1]), (((t + 1) / kSteps) & 1) ^ 1);
          }
        }
        mma_commit(smem_u32(&ctl->k_empty[st]));
        t_done = t + 1;
      }
      ctl->t_done = t_done;
    }
  } else if (warp >= 2 + kEpiThreads / 32) {
    // ---------------------------------------------------------------- scratch area, squared norms of the sampled rows
    const int at = threadIdx.x - (64 + kEpiThreads);
    if (at == 0) {
      // once some CTA has reported a timeout the rest of the grid winds down at once
      int poisoned = *reinterpret_cast<volatile int32_t*>(status);
      int slot = -1;
      if (kOnChip) {
        slot = 0;                             // (none needed)
      } else if ((int)gridDim.x <= p.slots) {
        slot = (int)blockIdx.x;               // an area for every CTA: nothing to search for
      } else {
        // a scratch area no resident CTA holds: there are as many as CTAs can be resident, so one is free; the
        // search starts at this SM's number and normally ends at once
        unsigned smid;
        asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
        for (int s = 0; s < 8 * p.slots && slot < 0; ++s) {
          const int cand = (int)((smid * kCtasPerSm + s) % (unsigned)p.slots);
          if (take_area(&p.slot_taken[cand])) slot = cand;
        }
        if (slot < 0) { atomicMin(status, (int32_t)COSA_ERR_DEVICE_TIMEOUT); poisoned = 1; }
      }
      ctl->slot = slot;
      ctl->poisoned = poisoned != 0;
      if (poisoned) ctl->abort_flag = 1;
      mbar_arrive(smem_u32(&ctl->slot_bar));
    }
    __syncwarp();
    auto wait_all = [&](uint32_t bar, uint32_t parity) { return kStrict ? mbar_poll_warp(bar, parity, abort_flag, budget) : mbar_wait_warp(bar, parity, abort_flag, budget); };
    float k2 = kOnChip ? 0.f : largest_key_norm(p, lane);
    bool alive = wait_all(smem_u32(&ctl->a_full), 0);
    if (alive && !kOnChip) {
#pragma unroll 1
      for (int row = at; row < kRows; row += kAuxThreads) ctl->q2[0][row] = norm2(smem + (size_t)(row / 128) * kTileBytes + (size_t)(row % 128) * 128, std::integral_constant<int, 16>{});
    }
    if (kOnChip) {
      // (a stage is not filled again before its keys' norms have been taken)
#pragma unroll 1
      for (int t = 0; t < n_tiles && alive; ++t) {
        alive = wait_all(smem_u32(&ctl->k_full[t % kStages]), (t / kStages) & 1);
        if (!alive) break;
#pragma unroll 1
        for (int row = at; row < 128; row += kAuxThreads) {
          const float s2 = norm2(smem + (size_t)kTileBytes * (kRowTiles + t % kStages) + row * 128, std::integral_constant<int, 16>{});
          if (s2 == s2 && t * 128 + row < ns_b) k2 = fmaxf(k2, s2);   // (a NaN row is left to the later stages; padding is no key)
        }
        if (kMedium) {
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&ctl->n_read[t % kStages]));
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) k2 = fmaxf(k2, __shfl_xor_sync(0xffffffffu, k2, o));
    }
    if (!alive && !*abort_flag) screen_timeout(ctl, status);
    if (lane == 0) ctl->k2w[at >> 5] = k2;
    __syncwarp();
    if (alive && lane == 0) mbar_arrive(smem_u32(&ctl->norm_bar));
  } else {
    // ---------------------------------------------------------------- kParts threads per sampled query row
    const int ew = warp - 2;
    const int sub = warp & 3;                // the TMEM lanes a warp may read: 32 * (warp % 4)
    const int rt = (ew >> 2) % kRowTiles;    // row tile
    const int part = ew / (4 * kRowTiles);   // column part
    const int row = rt * 128 + sub * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(sub * 32) << 16;
    const int grp = row / R, r = row % R;
    const int i = i0 + (grp >> lg), h = g * G + (grp & (G - 1));
    const bool row_ok = i < nqb_b;
    const int r_glob = i * R + r;                        // index among the head's sampled rows
    const int c_limit = p.causal ? r_glob : ns_b - 1;    // last sampled key this row may see
    constexpr int BPC = kPartCols / R;                   // key blocks per column part
    float top1 = -INFINITY, top2 = -INFINITY, top3 = -INFINITY;
    int jstar = 0, jstar2 = 0;
    // the CTA's block maxima: [tile][row group][block of the tile][row of the group], so that the R maxima one
    // score needs are contiguous
    constexpr int kTileFloats = kRows * BPT;
    const uint64_t keep = l2_policy_evict_last();
    // The epilogue warps meet at named barriers: every one of them comes, also after a wait that ran out, and all go on or none
    auto agree = [&](bool ok) { return !bar_red_or(1, kEpiThreads, !ok); };
    bool alive = wait_warp(smem_u32(&ctl->slot_bar), 0);
    if (!alive && !*abort_flag) screen_timeout(ctl, status);
    alive = alive && !ctl->poisoned;        // (set before the barrier completes: no lane sees it otherwise)
    if (kOnChip && alive) {                 // (nothing else to do until the first product is there)
      alive = wait_warp(smem_u32(&ctl->a_full), 0);
      if (!alive && !*abort_flag) screen_timeout(ctl, status);
      ctl->q2[part][row] = norm2(smem + (size_t)rt * kTileBytes + (size_t)(row % 128) * 128 + part * kHalfBytes, std::integral_constant<int, 8>{});
    }
    float* mine = p.maxima + (size_t)max(ctl->slot, 0) * ((size_t)((ns + 127) / 128) * kTileFloats) + ((size_t)grp * BPT + part * BPC) * R + r;
    // one key tile: this row's block maxima, and the three largest so far
    auto take_tile = [&](int t, float (&mb)[BPC]) {
      const int sb = t % kSteps, st = t % kStages;
      if (!wait_warp(smem_u32(&ctl->k_empty[st]), (t / kStages) & 1)) {   // this tile's MMAs finished
        if (!*abort_flag) screen_timeout(ctl, status);
        return false;
      }
      tc_fence_after();
      uint32_t v[kPartCols / 32][32];
#pragma unroll
      for (int c2 = 0; c2 < kPartCols / 32; ++c2)
        tmem_ld32(tmem + (sb * kRowTiles + rt) * 128 + lane_addr + part * kPartCols + c2 * 32, v[c2]);
      tmem_wait_ld();
      tc_fence_before();
      mbar_arrive(smem_u32(&ctl->s_empty[sb]));
#pragma unroll
      for (int bb = 0; bb < BPC; ++bb) {
        const int c0 = bb * R;                              // first column of the block within the part
        const int cabs = t * 128 + part * kPartCols + c0;   // ... and among the head's sampled keys
        float m0 = -INFINITY, m1 = -INFINITY;
        if (cabs + R - 1 <= c_limit) {                      // whole block visible: no masking
#pragma unroll
          for (int e = 0; e < R; e += 2) {
            m0 = fmaxf(m0, __uint_as_float(v[(c0 + e) / 32][(c0 + e) % 32]));
            m1 = fmaxf(m1, __uint_as_float(v[(c0 + e + 1) / 32][(c0 + e + 1) % 32]));
          }
        } else {
#pragma unroll
          for (int e = 0; e < R; ++e)
            if (cabs + e <= c_limit) m0 = fmaxf(m0, __uint_as_float(v[(c0 + e) / 32][(c0 + e) % 32]));
        }
        mb[bb] = fmaxf(m0, m1);
      }
      if (!kOnChip) {
        float* dst = mine + (size_t)t * kTileFloats;
#pragma unroll
        for (int bb = 0; bb < BPC; ++bb) st_l2_hint(dst + bb * R, mb[bb], keep);
      }
#pragma unroll
      for (int bb = 0; bb < BPC; ++bb) {
        const float m = mb[bb];
        const int jb = t * BPT + part * BPC + bb;
        // (selects, not branches: some lane of the warp inserts nearly always.  Stage 1 of 61 blocks 47.9 -> 45.5 us, of four prompts in
        // 16-token pages 164.8 -> 162, at 32K 167.5 -> 166.8; at 128K, where late tiles seldom hold a new maximum, 1,302 -> 1,308)
        const bool first = m > top1, second = m > top2;
        top3 = fmaxf(top3, fminf(m, top2));
        jstar2 = first ? jstar : (second ? jb : jstar2);
        top2 = fmaxf(top2, fminf(m, top1));
        jstar = first ? jb : jstar;
        top1 = fmaxf(top1, m);
      }
      return true;
    };
    float mb_all[kOnChip ? kMaxTiles : 1][BPC];
    if (kOnChip) {
      // (unrolled: the maxima are registers)
#pragma unroll
      for (int t = 0; t < kMaxTiles; ++t)
        if (t < n_tiles && alive) alive = take_tile(t, mb_all[t]);
    } else {
      for (int t = 0; t < n_tiles && alive; ++t) alive = take_tile(t, mb_all[0]);
    }
    if (alive) {
      // all tiles seen: merge the column parts' top-3 block maxima of every row
      ctl->xt[part][0][row] = top1; ctl->xt[part][1][row] = top2; ctl->xt[part][2][row] = top3;
      ctl->xj[part][0][row] = jstar; ctl->xj[part][1][row] = jstar2;
      alive = wait_warp(smem_u32(&ctl->norm_bar), 0);
      if (!alive && !*abort_flag) screen_timeout(ctl, status);
    }
    alive = agree(alive);
    if (alive) {
#pragma unroll
      for (int other = 1; other < kParts; ++other) {
        const int op = (part + other) % kParts;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const float m = ctl->xt[op][q][row];
          const int jb = q < 2 ? ctl->xj[op][q][row] : 0;
          if (m > top1) { top3 = top2; top2 = top1; jstar2 = jstar; top1 = m; jstar = jb; }
          else if (m > top2) { top3 = top2; top2 = m; jstar2 = jb; }
          else if (m > top3) top3 = m;
        }
      }
      // the row's best block, and whether the runner-up is too close to call
      // (the threshold grows with the magnitude of the row and of the call's keys, which is what the rounding error of a
      // logit follows)
      const float k2 = fmaxf(ctl->k2w[0], ctl->k2w[1]), q2 = kOnChip ? ctl->q2[0][row] + ctl->q2[1][row] : ctl->q2[0][row];
      static_assert(kAuxThreads == 64 && kParts == 2, "two aux warps, two halves");
      float g2 = q2;                                       // the group's rows are R consecutive lanes
#pragma unroll
      for (int o = 1; o < R; o <<= 1) g2 = fmaxf(g2, __shfl_xor_sync(0xffffffffu, g2, o));
      if (!kLists && part == 0 && r == 0 && row_ok) p.qk2max[(size_t)(b * p.hq + h) * p.nqb + i] = g2 * k2;
      const float tau_row = fmaxf(p.tau_row, 2.f * screen_error_bound(q2 * k2, p.scale));
      const bool amb = row_ok && (top1 - top2) * p.scale <= tau_row;
      const bool amb3 = row_ok && (top1 - top3) * p.scale <= tau_row;
      const unsigned any_amb = __ballot_sync(0xffffffffu, amb), any_amb3 = __ballot_sync(0xffffffffu, amb3);
      const int shift = (lane / R) * R;
      const unsigned grp_mask = (R == 32) ? 0xffffffffu : (((1u << R) - 1u) << shift);
      if (part == 0) {
        ctl->mstar[row] = top1;
        if (kLists) {
          ctl->j12[0][row] = jstar; ctl->j12[1][row] = jstar2;
          if (r == 0) { ctl->amb[grp] = (any_amb & grp_mask) >> shift; ctl->qk2[grp] = g2 * k2; ctl->hard[grp] = (any_amb3 & grp_mask) != 0; }
        }
        if (row_ok) {
          int2 js = make_int2(jstar, jstar2);
          reinterpret_cast<int2*>(p.jstar)[(size_t)(b * p.hq + h) * ns + r_glob] = js;
          if (r == 0) {
            p.ambmask[(size_t)(b * p.hq + h) * p.nqb + i] = (any_amb & grp_mask) >> shift;
            if (!kLists) p.hard[(size_t)(b * p.hq + h) * p.nqb + i] = (any_amb3 & grp_mask) ? 1 : 0;
          }
        }
      }
      if (kOnChip) {                // every product is done and every key read: the stages take the maxima
#pragma unroll
        for (int t = 0; t < kMaxTiles; ++t) {
          if (t < n_tiles) {
            float* dst = reinterpret_cast<float*>(smem + (size_t)kTileBytes * kRowTiles) + (size_t)t * kTileFloats + ((size_t)grp * BPT + part * BPC) * R + r;
#pragma unroll
            for (int bb = 0; bb < BPC; ++bb) dst[bb * R] = mb_all[t][bb];
          }
        }
      }
      // every row's M* in shared memory and every parked maximum visible to the whole CTA
      __threadfence_block();
      bar_sync(1, kEpiThreads);
      if (!kOnChip && threadIdx.x == 64) mbar_arrive(smem_u32(&ctl->parked_bar));
    }
    if (alive) {
      // block scores s_ij = sum over the group's rows of exp(M[r,j] - M*[r]) and HRM flags.  The parked maxima
      // come back through the key stages, which are idle by now: bulk copies of a stage's worth of tiles, several
      // in flight, by the producer (the fetch is a matter of latency, and no thread could hold that many bytes in registers);
      // one thread per (tile, row group, key block) then reads its R maxima from shared memory.
      constexpr int kOutsPerTile = kGroups * BPT;
      constexpr int kTileBytesM = kTileFloats * 4;
      constexpr int kTilesPerChunk = kTileBytes / kTileBytesM;
      static_assert(kTilesPerChunk >= 1 && kTileBytes % kTileBytesM == 0, "a stage holds whole tiles of maxima");
      const int et = threadIdx.x - 64;
      const int n_chunks = (n_tiles + kTilesPerChunk - 1) / kTilesPerChunk;
      const int oo = et % kOutsPerTile;
      const int blk = oo % BPT, og = oo / BPT;             // consecutive lanes: consecutive key blocks
      const int oi = i0 + (og >> lg), oh = g * G + (og & (G - 1));
      const int J = p.causal ? oi + 1 : nqb_b;
      const float kLog2e = 1.4426950408889634f;
      const float scale2 = p.scale * kLog2e;
      // a thread reads its R maxima as R/4 vectors, starting at a vector that depends on the lane so that the
      // lanes of a quarter warp hit different banks; M* is taken in the same rotated order
      constexpr int kVecs = R / 4;
      const int rot = (lane / (8 / kVecs > 0 ? 8 / kVecs : 1)) % kVecs;
      float nms[R];                                          // -M*
#pragma unroll
      for (int v4 = 0; v4 < kVecs; ++v4) {
        const int src = ((v4 + rot) % kVecs) * 4;
#pragma unroll
        for (int q = 0; q < 4; ++q) nms[v4 * 4 + q] = -ctl->mstar[og * R + src + q];
      }
      const unsigned long long scale22 = pack_f32x2(scale2, scale2);
      // (lists: the scores stay, in the third key stage behind the maxima, or where the query rows were; the keys come to the fourth, or
      // where the parked maxima were)
      constexpr int kCap = kLongLists ? kLongListCap : kListCap;
      static_assert(!kOnChip || (size_t)kMaxTiles * kTileFloats * 4 <= 2 * kTileBytes, "two stages hold the maxima");
      static_assert((size_t)kGroups * kListCap * 8 <= kTileBytes && (!kOnChip || !kLists || kMaxTiles * BPT <= kListCap), "a stage holds the keys of all lists");
      static_assert((size_t)kGroups * kLongListCap * 4 <= kRowTiles * kTileBytes && (size_t)kGroups * kLongListCap * 8 <= kStages * kTileBytes, "room for long lists");
      float* lists = reinterpret_cast<float*>(smem + (kLongLists ? 0 : (size_t)kTileBytes * (kRowTiles + 2)));
      float* srow = kLists ? lists + og * kCap : p.scores + ((size_t)(b * p.hq + oh) * p.nqb + min(oi, p.nqb - 1)) * p.nqb;
      // the score of tile tl's outputs that are this thread's, from the maxima at `maxima`
      auto score = [&](int tile, const float* maxima) {
        const int j = tile * BPT + blk;
        if (oi < nqb_b && j < J) {
          const float4* src = reinterpret_cast<const float4*>(maxima + ((size_t)og * BPT + blk) * R);
          unsigned long long sum = pack_f32x2(0.f, 0.f);         // (two sums, over even and odd rows)
          bool fl = false;
          // exp(M[r,j] - M*[r]) of two rows; 0 for invisible blocks
          auto two = [&](float x, float y, int r) {
            float u, v;
            unpack_f32x2(mul_f32x2(add_f32x2(pack_f32x2(x, y), pack_f32x2(nms[r], nms[r + 1])), scale22), u, v);
            sum = add_f32x2(sum, pack_f32x2(ex2_approx(u), ex2_approx(v)));
            fl = fl || x == -nms[r] || y == -nms[r + 1];
          };
#pragma unroll
          for (int v4 = 0; v4 < kVecs; ++v4) {
            const float4 x = src[(v4 + rot) % kVecs];
            two(x.x, x.y, v4 * 4);
            two(x.z, x.w, v4 * 4 + 2);
          }
          float e0, e1;
          unpack_f32x2(sum, e0, e1);
          const float e = e0 + e1;
          srow[j] = fl ? -e : e;                                 // sign bit carries the HRM flag
        }
      };
      if (kOnChip) {
        for (int o = et; o < n_tiles * kOutsPerTile; o += kEpiThreads) {
          const int tl = o / kOutsPerTile;
          score(tl, reinterpret_cast<const float*>(smem + (size_t)kTileBytes * kRowTiles) + (size_t)tl * kTileFloats);
        }
      }
      int c_done = 0;
      for (int c = 0; !kOnChip && c < n_chunks && alive; ++c) {
        const int st = c % kStages;
        alive = wait_warp(smem_u32(&ctl->m_full[st]), (c / kStages) & 1);
        if (!alive) { if (!*abort_flag) screen_timeout(ctl, status); break; }
        const int tiles_here = min(kTilesPerChunk, n_tiles - c * kTilesPerChunk);
        const float* stage = reinterpret_cast<const float*>(smem + (size_t)kTileBytes * (kRowTiles + st));
        for (int o = et; o < tiles_here * kOutsPerTile; o += kEpiThreads) {
          const int tl = o / kOutsPerTile;
          score(c * kTilesPerChunk + tl, stage + (size_t)tl * kTileFloats);
        }
        mbar_arrive(smem_u32(&ctl->m_empty[st]));
        c_done = c + 1;
      }
      if (et == 0) ctl->c_done = c_done;
      if (kLists) {
        // a warp per list
        alive = agree(alive);
        unsigned long long* keys = reinterpret_cast<unsigned long long*>(smem + (size_t)kTileBytes * (kRowTiles + (kLongLists ? 0 : 3)));
#pragma unroll 1
        for (int x = ew; x < kGroups && alive; x += kEpiThreads / 32) {
          const int li = i0 + (x >> lg), lh = g * G + (x & (G - 1));
          if (li >= nqb_b) break;
          const int cand = p.causal ? li + 1 : nqb_b;
          auto make = [&](auto per) {
            make_list<R, decltype(per)::value, !kLongLists>(kp, p, tau_score, b, g, lh, li, cand, ctl->amb[x], ctl->hard[x], ctl->qk2[x], lists + x * kCap,
                                                            &ctl->j12[0][x * R], &ctl->j12[1][x * R], keys + x * kCap, lane);
          };
          if (!kLongLists || cand <= 64) make(std::integral_constant<int, 2>{});
          else if (cand <= 128) make(std::integral_constant<int, kLongLists ? 4 : 2>{});
          else make(std::integral_constant<int, kLongLists ? 8 : 2>{});
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    // the kernel gave up somewhere: copies and products still in flight finish on their own and must have done so
    // before the CTA's shared and tensor memory go to the next one
    (void)mbar_wait_noabort(smem_u32(&ctl->a_full), 0);
    const int ti = ctl->t_issued, td = ctl->t_done;
    for (int tt = max(0, ti - kStages); tt < ti; ++tt) (void)mbar_wait_noabort(smem_u32(&ctl->k_full[tt % kStages]), (tt / kStages) & 1);
    if (td > 0) (void)mbar_wait_noabort(smem_u32(&ctl->k_empty[(td - 1) % kStages]), ((td - 1) / kStages) & 1);
    const int cf = ctl->c_fetched;
    for (int cc = max(ctl->c_done, cf - kStages); cc < cf; ++cc) (void)mbar_wait_noabort(smem_u32(&ctl->m_full[cc % kStages]), (cc / kStages) & 1);
  }
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, kTmemCols);
  if (kOnChip) return;
  {
    if (ctl->slot < 0) return;            // (the CTA has no area)
    // the parked maxima are dead: let L2 drop the lines instead of writing them back
    char* area = reinterpret_cast<char*>(p.maxima + (size_t)ctl->slot * ((size_t)((ns + 127) / 128) * (kRows * BPT)));
    const size_t bytes = (size_t)n_tiles * (kRows * BPT) * sizeof(float);
    for (size_t off = (size_t)threadIdx.x * 128; off < bytes; off += (size_t)kThreads * 128)
      asm volatile("discard.global.L2 [%0], 128;" ::"l"(area + off) : "memory");
  }
  if ((int)gridDim.x <= p.slots) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicExch(&p.slot_taken[ctl->slot], 0);
  }
}

}  // namespace

bool kap_screen_supported(int rows, int group, int stride, const KvPaging& pg) {
  if (!((rows == 8 || rows == 16 || rows == 32) && group * rows <= kRows && kRows % (group * rows) == 0)) return false;
  // paged keys: a page must hold at least 8 sampled rows (boxes land on 1024-byte boundaries of the swizzled tile)
  return !pg.table || pg.page_size / stride >= 8;
}

int kap_screen_grid(int batch, int hq, int hkv, int nqb, int stride) {
  const int QB = kRows / ((hq / hkv) * (128 / stride));
  return batch * hkv * ((nqb + QB - 1) / QB);
}

int kap_screen_slots() {
  return device_sm_count() * kCtasPerSm;
}

// Lists of up to kLongListCap candidates are made here (512 are 16 keys a lane, whose sort takes a warp four times as long as 8).  The
// medium form's 8 tiles would want 64 maxima a thread with 8 sampled rows a block.
ScreenForm kap_screen_form(const KapParams& p) {
  const int keys = p.n / p.stride;
  const bool is_short = keys <= 128 * kStages, lists = p.qtiles == 1 && p.sort_mode == 0 && p.nqb <= kLongListCap;
  if (is_short) return lists ? kScreenShortLists : kScreenShort;
  if (!lists) return kScreenLong;
  return p.rows >= 16 && keys <= 128 * kMediumTiles ? kScreenMediumLists : kScreenLongLists;
}

size_t kap_screen_slot_bytes(int n, int stride) {
  const size_t ns = (size_t)n / stride, R = 128 / stride;
  return ((ns + 127) / 128) * kRows * (128 / R) * sizeof(float);
}

cudaError_t launch_kap_screen(const KapParams& kp, const KapScreenParams& p_in, float tau_score, cudaStream_t st) {
  KapScreenParams p = p_in;
  const int R = 128 / p.stride;
  const ScreenForm form = kap_screen_form(kp);
  if (screen_parks(form) && (!p.maxima || !p.slot_taken || p.slots <= 0)) return cudaErrorInvalidValue;
  const uint64_t ns = (uint64_t)p.n / p.stride;
  CUtensorMap qm, km;
  // every `stride`-th row of q and k: the row stride of the maps is `stride` rows of the tensor (of the page pool)
  const int k_box = p.pg.table ? ((p.pg.page_size / p.stride) < 128 ? p.pg.page_size / p.stride : 128) : 128;
  const Strides qs = {p.qs.b, p.qs.h, p.qs.t * p.stride};
  // the heads of a group in one box, if rows lie inside heads (so that the box lays them out head by head) and 128 rows hold it
  const int group = p.hq / p.hkv;
  p.q_box_heads = group * R <= 128 ? group : 128 / R;
  bool ok = make_tile_map(&qm, &p.qo, p.q, ns, (uint64_t)p.hq, (uint64_t)p.batch, qs, R, p.q_box_heads);
  if (ok && p.qo.row > p.qo.head) {
    p.q_box_heads = 1;
    ok = make_tile_map(&qm, &p.qo, p.q, ns, (uint64_t)p.hq, (uint64_t)p.batch, qs, R);
  }
  if (p.pg.table) {
    const Strides pool = dense_strides(p.hkv, p.pg.page_size);
    ok = ok && make_tile_map(&km, &p.ko, p.k, (uint64_t)(p.pg.page_size / p.stride), (uint64_t)p.hkv, (uint64_t)p.pg.num_pages,
                             Strides{pool.b, pool.h, pool.t * p.stride}, k_box);
  } else {
    ok = ok && make_tile_map(&km, &p.ko, p.k, ns, (uint64_t)p.hkv, (uint64_t)p.batch, Strides{p.ks.b, p.ks.h, p.ks.t * p.stride}, k_box);
  }
  if (!ok) return cudaErrorInvalidValue;
  int32_t* status = device_status_word();
  if (!status) return cudaErrorInvalidSymbol;
  const int grid = kap_screen_grid(p.batch, p.hq, p.hkv, p.nqb, p.stride);
  p.n_iq = grid / (p.batch * p.hkv);
  p.group_shift = 0;
  while ((1 << p.group_shift) < group) ++p.group_shift;
  cudaError_t e;
#define COSA_LAUNCH_SCREEN(RR)                                                                                              \
  {                                                                                                                         \
    const bool strict = wait_budget_is_short(p.wait_budget);                                                                \
    constexpr int kMediumOr = RR >= 16 ? kScreenMediumLists : kScreenLongLists;                                              \
    auto pick = [&](auto strict_c) {                                                                                        \
      constexpr bool S = decltype(strict_c)::value;                                                                         \
      return form == kScreenShort ? kap_screen_kernel<RR, S, kScreenShort>                                                  \
           : form == kScreenShortLists ? kap_screen_kernel<RR, S, kScreenShortLists>                                        \
           : form == kScreenMediumLists ? kap_screen_kernel<RR, S, kMediumOr>                                               \
           : form == kScreenLongLists ? kap_screen_kernel<RR, S, kScreenLongLists> : kap_screen_kernel<RR, S, kScreenLong>; \
    };                                                                                                                      \
    auto kernel = strict ? pick(std::true_type{}) : pick(std::false_type{});                                                \
    static SmemLimit limits[10];                                                                                            \
    e = raise_smem_limit(reinterpret_cast<const void*>(kernel), &limits[2 * (int)form + (strict ? 1 : 0)], kScreenSmem);    \
    if (e != cudaSuccess) return e;                                                                                         \
    return launch_chained(kernel, dim3(grid), kThreads, kScreenSmem, st, qm, km, p, kp, tau_score, status);                               \
  }
  if (R == 8) { COSA_LAUNCH_SCREEN(8) }
  else if (R == 16) { COSA_LAUNCH_SCREEN(16) }
  else if (R == 32) { COSA_LAUNCH_SCREEN(32) }
  return cudaErrorInvalidValue;
#undef COSA_LAUNCH_SCREEN
}

}  // namespace cosa
