// OSK on the sm_100a tensor cores (Sec. 4.3; Algorithm A steps 7-21; skip rule Eq. 5).
//
// Two CTAs per SM, each walking one work item -- a (query head, query block) -- after another.  The walk of a work item is a
// chain of dependent steps -- K tile -> S = Q K_j^T -> row maxima -> tile vote -> (exponentials -> O += P V_j) -> next block
// -- and two independent walks fill each other's gaps.  An SM's resources are therefore halved: 256 columns of tensor memory,
// 113 KB of shared memory and 32 K registers per CTA, eight warps:
//   warps 0..3   one thread per query row: S row to registers, row maximum, vote, exponentials, P, epilogue
//   warp 4       K and V tiles ("physical jumping": only listed blocks are ever fetched)
//   warp 5       issues the products
//   warp 6       work items: takes them over, looks up their lists, fetches Q
//   warp 7       idle (warps 4 to 7 give registers to the first four)
// The running row maxima live in the threads' registers, the tile vote of Eq. (5) is one barrier, which only warps that would skip
// wait at, and every thread counts the computed blocks for itself: no exchange between warps beyond that barrier.
//
// Tensor memory has room for one S (128 columns) beside O (128); the second S buffer is the row threads' registers: they copy S
// out at once, and Q K^T of the next position runs while they work on this one, before it is known whether the block will be
// computed or skipped.  P therefore cannot lie over S: it goes to shared memory, 64 keys at a time (16 KB, what Q and two tile
// slots leave), so that the product of its first half runs while the exponentials of the second are formed.  With Stage 2 off the
// first half goes to tensor memory, into the columns S has left, and Q K^T of the next position follows the product on it: it
// has the second half's exponentials to run under, V's first half comes a position ahead, and neither half waits for the
// other's place (all blocks of 16K 2,009 -> 1,965 us, 64K at 12.5 % 4,232 -> 4,199; both halves there, S behind the
// whole block: 2,130 and 4,494).  Not with Stage 2 on, where S must not wait for a V tile that is asked for after the vote, and not
// with pages smaller than a key block: a tile of theirs is many copies, and K(k + 2) would be asked for later.  (32 keys at a time
// through the same buffer: 2 to 6 % slower, each hand-over costs the rows a proxy fence.)
// Tiles: two slots X and Y.  When block k is decided, X holds K(k+1) and Y is free or holds the last V tile.  Skipped: K(k+2)
// goes to Y, and the slots change roles.  Computed: V(k) goes to Y, each 64-key half as soon as the product on the half before
// it has released it, and K(k+2) to X when Q K^T of k+1 is done.
// Work items: the grid has one CTA per item, but a CTA that nears the end of its walk takes over one that has not been started
// (clusterlaunchcontrol).  A warp of its own decodes it and looks up its list while the walk before goes on (in the load warp that
// took 4,900 cycles between the last V tile and the next K tile); Q and K tiles follow when the last Q K^T has released theirs,
// and the next walk's first S is there when the rows have written the output.  With a CTA an item, start and end of a walk kept a
// CTA 11,000 cycles busy (barriers, tensor memory, list, first tiles, output, next CTA), three computed blocks' worth.  Asked too
// early, the last items are dealt out badly: at a walk's start, all blocks of 16K (walks of 1 to 128 blocks) take 3 % longer than
// when four positions are left.
// What runs once an item is cold in the instruction cache and costs by its size, and the loop of a computed block (some 22 KB over
// all roles) loses lines to it: 225 requests an item go to the next cache on walks of 3.4 blocks, 20 a block on long ones.  Code is
// therefore shared rather than unrolled or inlined twice where walks are short (a form of 88 KB instead of 61: 236 us instead of
// 209 on walks of 3.4 blocks; one place that fetches K and V tiles instead of two: 175 -> 169, and 3 % of the walks of four
// prompts in 16-token pages); with Stage 2 and with small pages long ones have it written out (kLongWalks).
// What bounds it: tensor pipe and exponentials both want about 1,024 cycles of an SM per computed block, 512 per skipped one.  By
// clock stamps an SM takes 1,600 cycles a computed block with Stage 2 off, 2,100 with it on (the vote, and V only after it), 620 a
// skipped one -- a product whose operands both come from shared memory takes the tensor pipe 570 to 600, not 512 -- and 2,600 a work
// item.  (Cycles of the SM's own counter, which runs at 1.65 to 1.75 GHz under this kernel even where 1,965 MHz are reported.)  At 32K
// tokens the pipe is busy 58 % of the time, shared memory's data pipe 82 % (operands 58, threads 24).  A walk alone on an SM takes
// 3,900 cycles a computed block: two fill each other's waits, the row threads of both together want 2,500 for two blocks.
// Single launches, 32 query heads: 128K tokens and 4 % computed 6.7 to 7.0 ms on four GPUs, 32K and 8 % 0.90, all blocks of 16K 1.74, walks of
// 3.4 blocks (2 x 7,808 tokens) 0.158 (with a CTA an item 7.51, 1.08, 1.92 and 0.246).
// Every wait is bounded; a wait that runs out sets the device status word and the CTA winds down without writing
// further results (a work item's are written whole or not at all): load and issue warps leave, the row threads, whom no wait holds any more, run to the end of their list.
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "ptx_sm100.cuh"
#include "tile_maps.cuh"

namespace cosa {
namespace {

using namespace ptx;

constexpr int kTileBytes = kBlock * kHeadDim * 2;  // 32 KiB: one 128 x 128 bf16 tile
constexpr int kHalfBytes = kTileBytes / 2;         // K: one TMA box, 128 rows x 64 columns.  V: 64 rows, two boxes.  P: 128 rows x 64 keys
constexpr int kQuarterBytes = kTileBytes / 4;      // V: one TMA box, 64 rows x 64 columns
constexpr int kHalfKeys = kBlock / 2;
constexpr int kThreads = 256;
constexpr int kCtasPerSm = 2;
constexpr int kTmemCols = 256;
constexpr int kLoadWarp = 4, kMmaWarp = 5, kItemWarp = 6;
constexpr int kAskAhead = 4;                       // positions (or two computed blocks) before a walk's end at which more work is asked for
constexpr int kShortWalk = 8, kShortWalkPages = 4;  // list pitch up to which walks count as short, with Stage 2 and, without it, with small pages
constexpr uint32_t kDecComputed = 1, kDecEnd = 2;
constexpr int kTimedOut = 1, kPoisoned = 2;

struct __align__(16) Item {        // a work item as the item warp hands it to the others
  int row;                         // (batch item * query heads + query head) * query blocks + query block; < 0: there are no more
  int cnt, cap;                    // listed blocks, computed blocks at which Stage 2 ends the walk
  float theta2;                    // ln(Delta / N) in base 2, -inf where the test is off
  int j0, j1;                      // the first two listed blocks
  long long out_at;                // element offset of the item's first output row
  int b, g, i;                     // batch item, KV head, query block
  int q;                           // which Q tile it is
};
static_assert(sizeof(Item) == 48, "three 16-byte reads");

struct __align__(16) Control {
  unsigned long long grant[2];     // the grid's answer to a request for another work item (16 bytes)
  unsigned long long grant_bar;    // it has come
  unsigned long long item_bar[2];  // the t-th work item (by parity of t) is in item[]
  unsigned long long item_read[2]; // ... and has been read by every role
  unsigned long long q_free;       // every Q K^T of a walk has finished
  unsigned long long q_full;       // the item's Q tile has landed
  unsigned long long k_full[2];    // K(k) has landed (by parity of k)
  unsigned long long v_full[2];    // by half: the n-th V tile's half has landed
  unsigned long long s_full;       // Q K^T of the position has finished
  unsigned long long s_first;      // the same for the first position of a walk (a waiter may come when the second has finished, too)
  unsigned long long s_read;       // (unless P goes over S) every row has taken its S to registers
  unsigned long long dec_bar[2];   // the decision of a position (by parity) is in dec[]
  unsigned long long p_full[2];    // by half: the n-th P's half is in shared memory (the first may be in tensor memory)
  unsigned long long pv_done[2];   // by half: the n-th product with that half has finished (one barrier each: a waiter may be
                                   // a whole block late, and one parity bit cannot tell two phases apart)
  unsigned long long fin;          // every product has finished
  uint32_t tmem_base;
  volatile int abort_flag;         // kTimedOut, kPoisoned
  volatile int first_k;            // the item warp has requested K(0)
  volatile int req[6];             // requested by the time the load warp left: K tiles by parity, V tiles by half, Q tiles, work items
  volatile int diag[2];            // K(k) (by parity of k) is the diagonal block
  volatile uint32_t dec[2];
  volatile int yes[3];             // the last position (by threes) that some row votes to compute
  Item item[2];
};

constexpr size_t kSmemBytes = (size_t)kTileBytes * 3 + kHalfBytes + sizeof(Control);
static_assert(kSmemBytes + 1024 <= 233472 / 2, "shared memory budget of one of two CTAs");


__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&t);
}

// Token-level causal mask of the diagonal block, on one warp's rows of S in tensor memory: of the first 32 * warp columns every row
// sees all, of the next 32 those up to its own.  (On the 128 registers the rows then hold it was 4 KB of selects, cold once a walk: 31
// blocks of 32 heads 38.1 -> 37.0 us, 2 x 61 blocks 169.2 -> 166.5, all blocks of 16K 1,838 -> 1,810.)
__device__ __forceinline__ void mask_diagonal(uint32_t s, int warp, int lane) {
  uint32_t v[32];
  tmem_ld32(s + warp * 32, v);
  tmem_wait_ld();
#pragma unroll
  for (int c = 0; c < 32; ++c) if (c > lane) v[c] = 0xff800000u;   // -inf
  tmem_st32(s + warp * 32, v);
  if (warp < 3) {
#pragma unroll
    for (int c = 0; c < 32; ++c) v[c] = 0xff800000u;
#pragma unroll 1
    for (int q = warp + 1; q < 4; ++q) tmem_st32(s + q * 32, v);
  }
  tmem_wait_st();
}

// kMask: walk a binary block mask instead of the order lists (see BlockWalk); a compile-time switch so that the
// list-driven kernel carries none of the walk's state
// kStage2: false = Stage 2 off (tightened_budget >= 1: Eq. 4, attention over the listed blocks; the library's dense
//          path): every listed block is computed, no vote is taken
// kSmallPages: K and V are page pools whose pages are smaller than a key block (Sec. C.1: a logical block resolved
//          through several physical pages).  A tile is then assembled from one pair of boxes per page, which the lanes
//          of the load warp issue side by side, each after its own table look-up.  Boxes land on 1024-byte boundaries of
//          the tile (pages of at least 8 tokens), where the 128-byte swizzle, a function of the shared-memory address,
//          gives the layout of the one-piece tile.
// kLongWalks: (Stage 2 or small pages) copies of the code that runs once a position or once an item are written out (see above); else they
//          are shared
template <bool kMask, bool kStage2, bool kSmallPages, bool kLongWalks>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
osk_tc_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
              const __grid_constant__ CUtensorMap v_map, OskParams p, int32_t* status) {
  constexpr bool kPInTmem = !kStage2 && !kSmallPages;   // P's first half goes to tensor memory, over S
  // Short walks: a CTA's first tile is asked for by the item warp (8 blocks of 2 heads 7.4 -> 6.9 us; whole passes enqueued ahead of the
  // device, medians of 25 within 0.1 to 0.3: 8 blocks of 2 heads 18.9 -> 18.5, 32 of 4 heads 27.1 -> 26.4, 31 of 32 heads 47.3 -> 47.0; with the
  // longer code 2 x 61 blocks +1.8 %, 32K +1.3)
  constexpr bool kEarlyTile = kStage2 && !kLongWalks && !kMask;
  extern __shared__ __align__(1024) unsigned char smem_raw[];   // swizzled tiles need 1024-byte alignment
  unsigned char* smem = smem_raw;
  const uint32_t base = smem_u32(smem_raw);
  if (base & 1023u) {   // never expected; refuse to run rather than compute on misplaced tiles
    if (threadIdx.x == 0) atomicMin(status, (int32_t)COSA_ERR_CUDA);
    return;
  }
  const uint32_t q_sm = base;
  const uint32_t x_sm = base + kTileBytes;          // the two tile slots
  const uint32_t p_sm = base + 3 * kTileBytes;      // 64 keys of P
  Control* ctl = reinterpret_cast<Control*>(smem + (size_t)kTileBytes * 3 + kHalfBytes);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (uniform, which the compiler cannot know)
  const int G = p.group;
  chain_wait();

  int b = 0, g = 0, i = 0;                 // (load warp, item warp) batch item, KV head, query block
  // (whole warp) part 0 or 1: that half of V's key block j to tile slot `slot`; part 2: K's key block j as tile K(k).  Box
  // after box: `box` bytes from one 64-column half of d to the other.  One lane arms the barrier; with small pages every lane then
  // fetches one page's part
  auto fetch = [&](int part, int j, int slot, int k) {
    const bool is_k = part == 2;
    const CUtensorMap* map = is_k ? &k_map : &v_map;
    const uint32_t bar = smem_u32(is_k ? &ctl->k_full[k & 1] : &ctl->v_full[part]);
    const uint32_t dst = x_sm + slot * kTileBytes + (part == 1 ? kHalfBytes : 0), box = is_k ? kHalfBytes : kQuarterBytes;
    const int row0 = j * kBlock + (part == 1 ? kHalfKeys : 0);
    auto part_of = [&](int at) {
      const KvCoord c = kv_coord(p.pg, b, g, row0 + at);
#pragma unroll
      for (int x = 0; x < 2; ++x)
        tma_load_tile(dst + x * box + at * 128, map, x * 64, c.row, c.head, c.outer, p.ko.row, p.ko.head, p.ko.outer, bar);
    };
    if (elect_one()) {
      if (is_k) ctl->diag[k & 1] = p.causal && j == i;
      mbar_expect_tx(bar, 2 * box);
      if (!kSmallPages) part_of(0);       // (a page holds whole key blocks)
    }
    if (kSmallPages) {
      __syncwarp();
      const int rows = is_k ? kBlock : kHalfKeys, ps = min(p.pg.page_size, rows), at = lane * ps;
      if (at < rows) part_of(at);
    }
  };
  // (item warp) work items: KV head major, then query blocks from the longest list down, the group's query heads innermost, so
  // that CTAs resident together read the same K/V pages
  int h = 0;
  auto decode = [&](int w) {
    const int bg = divided(w, p.by_kv), wk = w - bg * (G * p.nqb), back = divided(wk, p.by_group);
    b = divided(bg, p.by_hkv);
    g = bg - b * p.hkv;
    i = p.nqb - 1 - back;
    h = g * G + wk - back * G;
  };
  // its count, its first two list entries and the status word, one in each of the first lanes
  auto look_up = [&]() {
    const size_t row = (size_t)(b * p.hq + h) * p.nqb + i;
    int v = 0;
    if (lane == 3) v = *reinterpret_cast<volatile int32_t*>(status);   // once some CTA has reported a timeout no further work is begun
    else if (!kMask && lane == 0) v = p.count[row];
    else if (!kMask && lane < 3 && lane <= p.order_stride) v = p.order[row * p.order_stride + lane - 1];
    return v;
  };
  auto fetch_q = [&]() {                  // (one lane)
    mbar_expect_tx(smem_u32(&ctl->q_full), kTileBytes);
    tma_load_tile(q_sm, &q_map, 0, i * kBlock, h, b, p.qo.row, p.qo.head, p.qo.outer, smem_u32(&ctl->q_full));
    tma_load_tile(q_sm + kHalfBytes, &q_map, 64, i * kBlock, h, b, p.qo.row, p.qo.head, p.qo.outer, smem_u32(&ctl->q_full));
  };
  int head = 0;
  if (warp == kItemWarp) { decode(blockIdx.x); head = look_up(); }
  auto clamp_id = [&](int j) { return min(max(j, 0), p.nqb - 1); };

  if (warp == kItemWarp) {
    if (lane == 0) {
      mbar_init(smem_u32(&ctl->grant_bar), 1); mbar_init(smem_u32(&ctl->q_full), 1); mbar_init(smem_u32(&ctl->q_free), 1);
      for (int s = 0; s < 2; ++s) {
        mbar_init(smem_u32(&ctl->item_bar[s]), 1); mbar_init(smem_u32(&ctl->item_read[s]), kBlock + 2);
        mbar_init(smem_u32(&ctl->k_full[s]), 1); mbar_init(smem_u32(&ctl->v_full[s]), 1);
        mbar_init(smem_u32(&ctl->dec_bar[s]), 4); mbar_init(smem_u32(&ctl->p_full[s]), kStage2 ? kBlock : 4);
        mbar_init(smem_u32(&ctl->pv_done[s]), 1);
      }
      mbar_init(smem_u32(&ctl->s_full), 1); mbar_init(smem_u32(&ctl->s_first), 1); mbar_init(smem_u32(&ctl->s_read), kBlock);
      mbar_init(smem_u32(&ctl->fin), 1);
      ctl->abort_flag = 0; ctl->first_k = 0;
      for (int q = 0; q < 6; ++q) ctl->req[q] = 0;
      for (int q = 0; q < 3; ++q) ctl->yes[q] = -1;
      mbar_fence_init();
      fence_proxy_async_smem();
      // the first Q at once: its address needs nothing from global memory, while the list entries, the count and the status
      // word requested above are still on their way
      fetch_q();
    }
    __syncwarp();
  } else if (warp == kMmaWarp) {
    tmem_alloc(smem_u32(&ctl->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  chain_next();                            // (tensor memory is allocated)
  const uint32_t tmem_s = ctl->tmem_base, tmem_o = tmem_s + 128u;
  volatile int* abort_flag = &ctl->abort_flag;
  const long long budget = p.wait_budget;

  if (warp >= kLoadWarp) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    // (one answer per warp: all lanes fetch together)
    auto wait = [&](unsigned long long* bar, int phase) { return mbar_wait_warp(smem_u32(bar), phase & 1, abort_flag, budget); };
    // Further items come from the grid itself, in launch order, as long as CTAs of it are waiting for an SM.  (A grid that fits
    // on the chip asks for none: a CTA might take what an SM is about to start)
    const bool ask = (int)gridDim.x > p.wave;
    if (warp == kItemWarp) {
      // ---------------------------------------------------------------- work items, Q tiles
      // These waits last as long as a walk does, however short the steps of the others are: the caller's budget is theirs, and this
      // warp leaves when one of them has run out
      auto wait = [&](unsigned long long* bar, int phase) {
        return mbar_wait_warp(smem_u32(bar), phase & 1, abort_flag, max(budget, 1LL << 31));
      };
      int n_q = 1, n_walk = 0;                 // Q tiles requested (the first above), items with blocks
      int b_known = -1, nqb_b = 0;             // batch item of the lengths below
      float theta2 = -INFINITY;
      bool alive = true, more = true;
      for (int t = 0;; ++t) {
        const int raw_cnt = __shfl_sync(0xffffffffu, head, 0);
        int j0 = __shfl_sync(0xffffffffu, head, 1), j1 = __shfl_sync(0xffffffffu, head, 2);
        if (__shfl_sync(0xffffffffu, head, 3) != 0) {
          more = false;
          if (t == 0) *abort_flag = kPoisoned; // (Q has been requested for nothing)
        }
        int cnt = 0, cap = 0;
        if (more) {
          if (b != b_known) {
            b_known = b;
            nqb_b = item_blocks(p.pg, b, p.nqb);   // the item's own length in blocks; query blocks past it are padding
            // The CTA's first tile at once: by way of the load warp, whose code is cold, it is asked for 1,800 cycles later
            if (kEarlyTile && t == 0 && raw_cnt > 0 && i < nqb_b) {
              fetch(2, clamp_id(j0), 0, 0);
              if (lane == 0) ctl->first_k = 1;
            }
            // a batch item no longer than Delta would have ln(Delta/N) >= 0 and lose even its first block: the test is off for it
            const float th = p.use_threshold ? item_theta(p.pg, b, p.theta, p.skip_scale, nqb_b) : 0.f;
            theta2 = th < 0.f ? th * 1.4426950408889634f : -INFINITY;
          }
          const int J = p.causal ? i + 1 : max(nqb_b, 1);
          if (kMask) {
            BlockWalk walk;
            walk.init(p, (size_t)(b * p.hq + h) * p.nqb + i, J);
            cnt = i >= nqb_b ? 0 : min(walk.kept(), p.order_stride);
          } else {
            cnt = i >= nqb_b ? 0 : max(0, min(raw_cnt, p.order_stride));
          }
          cap = p.stage2 ? min(cnt, budget_count_fx(p.cap_fx, J)) : cnt;
        }
        if (t >= 2) alive = wait(&ctl->item_read[t & 1], (t >> 1) - 1);   // the item before the last has been read
        if (!alive) break;
        const bool next_q = cnt > 0 && t > 0;
        if (lane == 0) {
          Item* it = &ctl->item[t & 1];
          it->row = more ? (b * p.hq + h) * p.nqb + i : -1;
          it->cnt = cnt; it->cap = cap; it->theta2 = theta2; it->j0 = j0; it->j1 = j1;
          it->out_at = more ? elem_off(p.os, b, h, i * kBlock) : 0;
          it->b = b; it->g = g; it->i = i; it->q = next_q ? n_q : n_q - 1;
          mbar_arrive(smem_u32(&ctl->item_bar[t & 1]));
        }
        if (!more) break;
        if (next_q) {                           // its tile is free when the last Q K^T of the walk before has finished
          if (n_walk > 0) alive = wait(&ctl->q_free, n_walk - 1);
          if (!alive) break;
          if (elect_one()) fetch_q();
          ++n_q;
        } else if (t == 0 && cnt == 0) {
          alive = wait(&ctl->q_full, 0);        // (requested before the count was known)
          if (!alive) break;
        }
        if (cnt > 0) ++n_walk;
        more = false;
        if (ask) {
          alive = wait(&ctl->grant_bar, t);
          if (!alive) break;
          const int w2 = granted_work(smem_u32(ctl->grant));
          more = w2 >= 0;
          head = 0;
          if (more) { decode(w2); head = look_up(); }
        }
      }
      if (lane == 0) {
        if (!alive && !*abort_flag) *abort_flag = kTimedOut;
        ctl->req[4] = n_q;
      }
    } else if (warp == kLoadWarp) {
      // ---------------------------------------------------------------- tiles
      // Counters run on from walk to walk, as the barriers' phases do: tiles K(k), positions decided, blocks computed before
      // this walk.  All roles count alike.
      BlockWalk walk;                          // (kMask only)
      int n_k = 0, n_v = 0, n_grant = 0;       // requested
      int n_walk = 0;                          // items with blocks
      int y = 0;                               // slot that takes the next V tile (or K tile after a skipped block)
      bool v_in_y = false;                     // slot y holds, or held last, the V tile of the last computed block
      int k_base = 0, pos_base = 0, n_base = 0;
      bool alive = true;
      for (int t = 0; alive; ++t) {
        alive = wait(&ctl->item_bar[t & 1], t >> 1);
        if (!alive) break;
        const uint32_t at = smem_u32(&ctl->item[t & 1]);
        const uint4 f0 = ld_shared_128(at), f1 = ld_shared_128(at + 16), f2 = ld_shared_128(at + 32);
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&ctl->item_read[t & 1]));
        const int row = (int)f0.x, cnt = (int)f0.y, cap = (int)f0.z;
        if (row < 0) break;
        b = (int)f2.x; g = (int)f2.y; i = (int)f2.z;
        const int n_pos = cap > 1 ? cnt : min(cnt, 1);   // positions the walk can reach (the first block is always computed: with a cap of 1 the walk ends there)
        bool asked = !ask;
        auto request = [&]() {
          asked = true;
          ++n_grant;
          if (lane == 0) {
            fence_proxy_async_smem();
            mbar_expect_tx(smem_u32(&ctl->grant_bar), 16);
            request_work(smem_u32(ctl->grant), smem_u32(&ctl->grant_bar));
          }
        };
        if (n_pos > 0) {
          // key blocks of positions k, k + 1 and k + 2 (the last one requested a turn ahead), k starting at -2
          int j0 = 0, j1 = 0, j2 = (int)f1.x, j3 = (int)f1.y;
          if (kMask) {
            walk.init(p, (size_t)row, p.causal ? i + 1 : max(item_blocks(p.pg, b, p.nqb), 1));
            j2 = walk.at(0);
            j3 = cnt > 1 ? walk.at(1) : 0;
          }
          // slot y is free when the last Q K^T of the walk before has finished
          if (k_base > 0) alive = wait(&ctl->s_full, k_base - 1);
          const int32_t* list = p.order + (size_t)row * p.order_stride;   // unused when kMask
          // Turn k fetches V(k) and K(k + 2); turns -2 and -1: the first two K tiles, K(1) to the slot of the last V tile of the walk
          // before
          int k = -2, n = 0;                    // n: computed blocks before position k
          const bool v_before = v_in_y;
          v_in_y = false;
          while (alive) {
            uint32_t d = 0;
            if (k >= 0) {
              d = kDecComputed | (k == cnt - 1 ? kDecEnd : 0u);
              if (k == 0 && t == 0) {
                // (polled: a budget of a few cycles must run out here, see cosa_options.wait_cycles, and the wait is long)
                alive = mbar_poll_warp(smem_u32(kStage2 ? &ctl->dec_bar[0] : &ctl->s_first), 0, abort_flag, budget);
              } else if (kStage2 || k == 0) {
                alive = wait(kStage2 ? &ctl->dec_bar[(pos_base + k) & 1] : &ctl->s_first, kStage2 ? (pos_base + k) >> 1 : n_walk);
              }
              if (kStage2) d = ctl->dec[(pos_base + k) & 1];
            }
            const bool computed = (d & kDecComputed) != 0;
            // parts 0 and 1: the halves of V(k), each into a place that the product before has released; part 2: K(k + 2), into that of
            // K(k + 1) or of the last V tile
            const bool want_k = !(d & kDecEnd) && k + 2 < n_pos;
            auto do_part = [&](int part) {
              const bool is_k = part == 2, after_qk = is_k && computed;
              if (after_qk || (is_k && k == -1 ? v_before : v_in_y))
                alive = wait(after_qk ? &ctl->s_full : &ctl->pv_done[is_k ? 1 : part], after_qk ? k_base + k + 1 : n_base + n - 1);
              if (!alive) return;
              if (is_k) ++n_k; else ++n_v;
              if (!kEarlyTile || t > 0 || k > -2) fetch(part, clamp_id(is_k ? j2 : j0), is_k && (computed || k == -1) ? y ^ 1 : y, k_base + k + 2);   // (else: by the item warp)
            };
            if (kPInTmem) {
              // V(0)'s first half, V(k)'s second, V(k + 1)'s first (a turn ahead: its place is free before Q K^T of the next position begins),
              // K(k + 2)
#pragma unroll 1
              for (int step = k < 0 ? 3 : (k == 0 ? 0 : 1); step < 4; ++step) {
                const bool is_k = step == 3;
                if (is_k ? !want_k : step == 2 && (d & kDecEnd)) continue;
                const int at = step == 0 ? 0 : k + step - 1;       // (V) whose tile it is
                const bool after_qk = is_k && computed;
                if (is_k ? after_qk || (k == -1 && v_before) : at > 0)
                  alive = wait(after_qk ? &ctl->s_full : &ctl->pv_done[is_k || step == 1 ? 1 : 0], after_qk ? k_base + k + 1 : n_base + (is_k ? n : at) - 1);
                if (!alive) break;
                if (is_k) ++n_k; else ++n_v;
                fetch(is_k ? 2 : step & 1, clamp_id(is_k ? j2 : (step == 2 ? j1 : j0)), is_k && (computed || k == -1) ? y ^ 1 : y, k_base + k + 2);
              }
            } else if (!kLongWalks) {
#pragma unroll 1
              for (int part = computed ? 0 : 2; alive && part < (want_k ? 3 : 2); ++part) do_part(part);
            } else {
              if (computed) { do_part(0); if (alive) do_part(1); }
              if (alive && want_k) do_part(2);
            }
            if (!alive) break;
            if (!asked && (k + kAskAhead >= n_pos || n + 2 >= cap)) request();
            if (computed) { v_in_y = true; ++n; }
            if (d & kDecEnd) break;
            if (k >= 0 && !computed) { v_in_y = false; y ^= 1; }
            j0 = j1; j1 = j2; j2 = j3;
            if (k + 4 < n_pos) j3 = kMask ? walk.at(k + 4) : list[k + 4];
            ++k;
          }
          k_base += min(k + 2, n_pos); pos_base += k + 1; n_base += n;
          ++n_walk;
          y ^= 1;                               // (v_in_y: of the slot that is y ^ 1 from here on)
        }
        if (alive && !asked) request();
      }
      if (lane == 0) {
        if (!alive && !*abort_flag) *abort_flag = kTimedOut;
        ctl->req[0] = (n_k + 1) / 2; ctl->req[1] = n_k / 2; ctl->req[2] = (n_v + 1) / 2; ctl->req[3] = n_v / 2; ctl->req[5] = n_grant;
      }
    } else if (warp == kMmaWarp && elect_one()) {
      // ---------------------------------------------------------------- products
      auto wait = [&](unsigned long long* bar, int phase) { return mbar_wait(smem_u32(bar), phase & 1, abort_flag, budget); };
      const uint32_t idesc_qk = idesc_bf16(kBlock, kBlock, 0, 0);    // Q [M x K], K_j [N x K], both K-major
      const uint32_t idesc_pv = idesc_bf16(kBlock, kHeadDim, 0, 1);  // P [M x K] K-major, V_j [K x N] N-major
      const uint64_t qdesc = smem_desc_sw128(q_sm, 16, 1024), kdesc0 = smem_desc_sw128(x_sm, 16, 1024);
      const uint64_t pdesc = smem_desc_sw128(p_sm, 16, 1024), vdesc0 = smem_desc_sw128(x_sm, kQuarterBytes, 1024);
      auto issue_qk = [&](int k, int slot) {      // S = Q K^T with the k-th K tile
        if (!wait(&ctl->k_full[k & 1], k >> 1)) return false;
        tc_fence_after();
        mma_ss_x8<2, 4, 6, kHalfBytes / 16, kHalfBytes / 16 + 2, kHalfBytes / 16 + 4, kHalfBytes / 16 + 6>(
            tmem_s, qdesc, kdesc0 + (uint64_t)(slot * (kTileBytes / 16)), idesc_qk);
        mma_commit(smem_u32(&ctl->s_full));
        return true;
      };
      int y = 0, k_base = 0, pos_base = 0, n_base = 0;   // as in the load warp
      bool alive = true;
      for (int t = 0;; ++t) {
        alive = wait(&ctl->item_bar[t & 1], t >> 1);
        if (!alive) break;
        const uint32_t at = smem_u32(&ctl->item[t & 1]);
        const uint4 f0 = ld_shared_128(at);
        const int q = (int)ld_shared_128(at + 32).w;
        mbar_arrive(smem_u32(&ctl->item_read[t & 1]));
        const int cnt = (int)f0.y, n_pos = (int)f0.z > 1 ? cnt : min(cnt, 1);
        if ((int)f0.x < 0) break;
        if (n_pos == 0) continue;
        alive = wait(&ctl->q_full, q);
        int k = -1, n = 0;
        while (alive) {
          if (kPInTmem && k < 0 && n_base > 0) alive = wait(&ctl->pv_done[0], n_base - 1);   // (the walk before: P lay in S's place)
          if (!kPInTmem && k >= 0) alive = wait(&ctl->s_read, pos_base + k);
          if (alive && (!kPInTmem || k < 0) && k + 1 < n_pos) alive = issue_qk(k_base + k + 1, k < 0 ? y : y ^ 1);
          if (k < 0) {
            if (!kStage2 && alive) mma_commit(smem_u32(&ctl->s_first));
            ++k;
            continue;
          }
          uint32_t d = kDecComputed | (k == cnt - 1 ? kDecEnd : 0u);
          if (kStage2 && alive) {
            alive = wait(&ctl->dec_bar[(pos_base + k) & 1], (pos_base + k) >> 1);
            d = ctl->dec[(pos_base + k) & 1];
          }
          if (!alive) break;
          if (d & kDecEnd) mma_commit(smem_u32(&ctl->q_free));   // (Q K^T of a position that is not reached included)
          if (d & kDecComputed) {
#pragma unroll 1
            for (int half = 0; half < 2 && alive; ++half) {
              alive = wait(&ctl->v_full[half], n_base + n) && wait(&ctl->p_full[half], n_base + n);
              if (!alive) break;
              tc_fence_after();
              if (kPInTmem && half == 0) {           // P's first half lies in S's place: the next S behind its product
                mma_ts_x4<128, 256, 384>(tmem_o, tmem_s, vdesc0 + (uint64_t)(y * kTileBytes / 16), idesc_pv, n > 0);
                mma_commit(smem_u32(&ctl->pv_done[0]));
                if (k + 1 < n_pos) alive = wait(&ctl->pv_done[0], n_base + n) && issue_qk(k_base + k + 1, y ^ 1);
                continue;
              }
              // 16 keys per MMA: 32 bytes of a P row, 2 KiB (two 8-key groups) of the V half
              mma_ss_x4<2, 4, 6, 128, 256, 384>(tmem_o, pdesc, vdesc0 + (uint64_t)((y * kTileBytes + half * kHalfBytes) / 16), idesc_pv,
                                                n + half > 0);
              mma_commit(smem_u32(&ctl->pv_done[half]));
            }
            ++n;
          } else if (!(d & kDecEnd)) {
            y ^= 1;
          }
          if (d & kDecEnd) break;
          ++k;
        }
        if (!alive) break;
        k_base += min(k + 2, n_pos); pos_base += k + 1; n_base += n;
        y ^= 1;
      }
      if (!alive && !*abort_flag) *abort_flag = kTimedOut;
      mma_commit(smem_u32(&ctl->fin));                // also after a walk that was given up: tensor memory is released behind it
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
    // ------------------------------------------------------------------ one thread per query row
    const int r = threadIdx.x;                // query row inside the tile
    const uint32_t lane_addr = (uint32_t)(warp * 32) << 16;
    const float scale2 = p.scale * 1.4426950408889634f;   // work in base 2: exp(x) = exp2(x * log2 e)
    const int dec_words = (p.order_stride + 31) / 32;
    bool bad = false;                         // a wait of this thread ran out
    auto wait = [&](unsigned long long* bar, int phase) {
      if (!mbar_wait(smem_u32(bar), phase & 1, abort_flag, budget)) {
        bad = true;
        if (!*abort_flag) *abort_flag = kTimedOut;
      }
    };
    int k_base = 0, pos_base = 0, n_base = 0; // as in the load warp
    int turn = 0;                             // of the vote's barriers
    for (int t = 0;; ++t) {
      wait(&ctl->item_bar[t & 1], t >> 1);
      if (bar_red_or(1, kBlock, bad || *abort_flag)) break;
      const uint32_t at = smem_u32(&ctl->item[t & 1]);
      const uint4 f0 = ld_shared_128(at), f1 = ld_shared_128(at + 16);
      mbar_arrive(smem_u32(&ctl->item_read[t & 1]));
      const int cnt = (int)f0.y, cap = (int)f0.z;
      const float theta2 = __uint_as_float(f0.w);
      if ((int)f0.x < 0) break;
      const size_t row = f0.x;
      const size_t lse_at = row * kBlock + r;
      __nv_bfloat16* const out_tile = p.out + (long long)(((unsigned long long)f1.w << 32) | f1.z);
      if (cnt == 0) {
        // an empty list (not produced by KAP except for padding): zero output, nothing visited
        uint4 z = make_uint4(0, 0, 0, 0);
        uint4* dst = reinterpret_cast<uint4*>(out_tile + r * p.os.t);
#pragma unroll 1
        for (int c = 0; c < kHeadDim / 8; ++c) dst[c] = z;
        if (p.lse) p.lse[lse_at] = -INFINITY;
        if (r == 0) {
          if (p.visited) p.visited[row] = 0;
          if (p.scored) p.scored[row] = 0;
        }
        continue;
      }
      float m = -INFINITY;                      // running row maximum (base 2)
      float l = 0.f;                            // row sum
      int n = 0, kk = 0;                        // computed blocks, list position
      uint32_t dec_word = 0;
      uint32_t s[kBlock];                       // this row's raw logits, then probabilities
      for (;; ++kk) {
        wait(&ctl->s_full, k_base + kk);
        __syncwarp();
        tc_fence_after();
        if (ctl->diag[(k_base + kk) & 1]) mask_diagonal(tmem_s + lane_addr, warp, lane);
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(tmem_s + lane_addr + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&s[c * 32]));
        tmem_wait_ld();
        tc_fence_before();
        if (!kPInTmem) mbar_arrive(smem_u32(&ctl->s_read));
        // (three-input maxima: half the instructions of the two-input form)
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int c = 0; c < kBlock; c += 8) {
#pragma unroll
          for (int u = 0; u < 4; ++u) mx[u] = max3(mx[u], __uint_as_float(s[c + 2 * u]), __uint_as_float(s[c + 2 * u + 1]));
        }
        const float m_loc = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * scale2;   // scale > 0 commutes with max
        const float m_new = fmaxf(m, m_loc);
        bool last = kk == cnt - 1;
        if (kStage2) {
          // Eq. (5): skip iff max over the 128 rows of (m_loc - m) < ln(Delta/N), m including this block.  (Rows of a walk that was given
          // up vote on as long as their list lasts: nothing holds them any more)
          // A warp that votes to compute knows the outcome and goes on to its exponentials; the others wait for it.  Three barriers take
          // turns: Q K^T of the next position waits until every row has read S, so no warp votes twice ahead of another, and a warp whose
          // wait has run out goes on with the others only.  (All four at one barrier, an OR over its threads: 32K tokens 1,058 ->
          // 1,045 us, 128K 8,029 -> 7,955, walks of 3.4 blocks 179 -> 176, of 2 blocks 33.3 -> 32.5, 4K of 4 heads 14.4 -> 13.7)
          const int pos = pos_base + kk;
          bool compute = __any_sync(0xffffffffu, !((m_loc - m_new) < theta2));
          if (compute) ctl->yes[turn] = pos;
          if (compute && !__any_sync(0xffffffffu, bad)) {
            bar_arrive(2 + turn, kBlock);
          } else {
            bar_sync(2 + turn, kBlock);
            compute = ctl->yes[turn] == pos;
          }
          turn = turn == 2 ? 0 : turn + 1;
          last = last || n + (compute ? 1 : 0) == cap;
          ctl->dec[pos & 1] = (compute ? kDecComputed : 0u) | (last ? kDecEnd : 0u);
          mbar_arrive_if(smem_u32(&ctl->dec_bar[pos & 1]), lane == 0);
          if (p.decisions) {
            if (compute) dec_word |= 1u << (kk & 31);
            if ((kk & 31) == 31 || last) {
              if (r == 0 && !*abort_flag) p.decisions[row * dec_words + (kk >> 5)] = dec_word;
              dec_word = 0;
            }
          }
          if (!compute) {                           // skipped: nothing is added to l or O, and no maximum has moved
            if (last) break;
            continue;
          }
        }
        const float alpha = ex2_approx(m - m_new);  // (the first block: m = -inf)
        m = m_new;
        const bool moved = n > 0 && __any_sync(0xffffffffu, alpha != 1.f);
        // ---- P = exp(S - m), row sums (two elements per FMA and per add: the packed float32 forms), 64 keys at a time.
        // m is the maximum up to this block, so that an element that raises it weighs exactly 1 in bf16, and O is rescaled
        // whenever it moves.  (Left until it has moved by 2^8, a pass is 2 % faster, but the largest weights are rounded: error
        // against double precision over all blocks of 16K tokens 2.115e-3 instead of 2.016e-3, largest 6.6e-3 instead of 4.3e-3)
        l *= alpha;
        const unsigned long long sc2 = pack_f32x2(scale2, scale2), nm2 = pack_f32x2(-m, -m);
        unsigned long long acc01 = pack_f32x2(0.f, 0.f), acc23 = acc01;
        unsigned char* prow = smem + 3 * kTileBytes + r * 128;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          // the buffer's last reader: the second half of the block before, the first half of this one (asked now, needed
          // after the exponentials).  With the first half in tensor memory only second halves lie there, and O may be rescaled behind the
          // last product
          const int last_n = n_base + n - 1 + (kPInTmem ? 0 : half);
          unsigned long long* last_reader = &ctl->pv_done[kPInTmem ? 1 : half ^ 1];
          const bool is_free = (kPInTmem ? n == 0 || (half == 0 && !moved) : n + half == 0) || mbar_test_wait(smem_u32(last_reader), last_n & 1);
#pragma unroll
          for (int c = half * kHalfKeys; c < (half + 1) * kHalfKeys; c += 4) {
            float e0, e1, e2, e3;
            unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[c]), __uint_as_float(s[c + 1])), sc2, nm2), e0, e1);
            unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[c + 2]), __uint_as_float(s[c + 3])), sc2, nm2), e2, e3);
            e0 = ex2_approx(e0); e1 = ex2_approx(e1); e2 = ex2_approx(e2); e3 = ex2_approx(e3);
            acc01 = add_f32x2(acc01, pack_f32x2(e0, e1));
            acc23 = add_f32x2(acc23, pack_f32x2(e2, e3));
            s[c / 2] = pack_bf16(e0, e1); s[c / 2 + 1] = pack_bf16(e2, e3);
          }
          if (!is_free) wait(last_reader, last_n);
          if (half == 0 && moved) {                 // O = diag(alpha) O: the last product on it is the buffer's last reader
            __syncwarp();
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
              uint32_t o[32];
              tmem_ld32(tmem_o + lane_addr + c * 32, o);
              tmem_wait_ld();
#pragma unroll
              for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
              tmem_st32(tmem_o + lane_addr + c * 32, o);
            }
            tmem_wait_st();
          }
          if (kPInTmem && half == 0) {
            __syncwarp();
            tmem_st32(tmem_s + lane_addr, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
            tmem_wait_st();
          } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const uint32_t* e = &s[half * 32 + c * 4];
              *reinterpret_cast<uint4*>(prow + ((c ^ (r & 7)) << 4)) = make_uint4(e[0], e[1], e[2], e[3]);
            }
            fence_proxy_async_smem();
          }
          if (half == 0) tc_fence_before();         // (a rescaled O)
          // (one arrival a warp: all blocks of 16K 1,947 -> 1,924 us; with Stage 2 on equal, every thread arrives)
          if (!kStage2) __syncwarp();
          mbar_arrive_if(smem_u32(&ctl->p_full[half]), kStage2 || lane == 0);
        }
        {
          float r0, r1, r2, r3;
          unpack_f32x2(acc01, r0, r1);
          unpack_f32x2(acc23, r2, r3);
          l += (r0 + r1) + (r2 + r3);
        }
        ++n;
        if (last) break;
      }
      // ---- epilogue: the last product, then O / l as bf16.  The next walk's Q and K tiles are on their way meanwhile; the rows
      // of a warp go out through the warp's own rows of P, 64 columns at a time, so that a store covers whole 128-byte lines
      n_base += n;
      const float lse = (m + log2f(l)) * 0.6931471805599453f;
      wait(&ctl->pv_done[1], n_base - 1);
      const int n_pos = cap > 1 ? cnt : 1, n_issued = min(kk + 2, n_pos);   // (Q K^T of a position that was not reached: done, too)
      k_base += n_issued; pos_base += kk + 1;
      // (all rows agree whether the walk was given up: a work item is written whole or not at all)
      if (bar_red_or(1, kBlock, bad || *abort_flag)) break;
      tc_fence_after();
      const float inv = l > 0.f ? __frcp_rn(l) : 0.f;
      const unsigned long long inv2 = pack_f32x2(inv, inv);
      unsigned char* stage = smem + 3 * kTileBytes + warp * 4096;
      __nv_bfloat16* out = out_tile + (warp * 32 + (lane >> 3)) * p.os.t + (lane & 7) * 8;
      const long long out_step = 4 * p.os.t;
#pragma unroll (kLongWalks ? 2 : 1)
      for (int half = 0; half < 2; ++half) {
        uint32_t o[64];
        tmem_ld32(tmem_o + lane_addr + half * 64, *reinterpret_cast<uint32_t(*)[32]>(&o[0]));
        tmem_ld32(tmem_o + lane_addr + half * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&o[32]));
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          uint32_t pk[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float lo, hi;
            unpack_f32x2(mul_f32x2(pack_f32x2(__uint_as_float(o[c * 8 + 2 * e]), __uint_as_float(o[c * 8 + 2 * e + 1])), inv2), lo, hi);
            pk[e] = pack_bf16(lo, hi);
          }
          *reinterpret_cast<uint4*>(stage + lane * 128 + ((c ^ (lane & 7)) << 4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        }
        __syncwarp();
        uint4 piece[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {         // four rows, eight lanes a row
          const int rr = c * 4 + (lane >> 3);
          piece[c] = *reinterpret_cast<const uint4*>(stage + rr * 128 + (((lane & 7) ^ (rr & 7)) << 4));
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) *reinterpret_cast<uint4*>(out + c * out_step + half * 64) = piece[c];
        __syncwarp();
      }
      tc_fence_before();
      __syncwarp();
      if (p.lse) p.lse[lse_at] = lse;
      if (r == 32) {
        if (p.visited) p.visited[row] = n;
        if (p.scored) p.scored[row] = kk + 1;
        if (!kStage2 && p.decisions)
          for (int wd = 0; wd * 32 < cnt; ++wd) p.decisions[row * dec_words + wd] = cnt - wd * 32 >= 32 ? 0xffffffffu : ((1u << (cnt - wd * 32)) - 1u);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // A walk that was given up: products and copies in flight finish on their own and must have done so before the CTA
    // retires.  (Otherwise everything fetched has been waited for: Q K^T of the position after the last takes its tile, too.)
    if (threadIdx.x == 0) {
      if (*abort_flag == kTimedOut) atomicMin(status, (int32_t)COSA_ERR_DEVICE_TIMEOUT);
#pragma unroll 1
      for (int q = 0; q < 6; ++q) {
        unsigned long long* bar = q < 2 ? &ctl->k_full[q] : (q < 4 ? &ctl->v_full[q - 2] : (q == 4 ? &ctl->q_full : &ctl->grant_bar));
        const int c = kEarlyTile && q == 0 ? max(ctl->req[0], ctl->first_k) : ctl->req[q];
        if (c > 0) (void)mbar_wait_noabort(smem_u32(bar), (c - 1) & 1);
      }
      (void)mbar_wait_noabort(smem_u32(&ctl->fin), 0);
    }
    __syncthreads();
  }
  if (warp == kMmaWarp) tmem_dealloc(tmem_s, kTmemCols);
}

}  // namespace

cudaError_t launch_osk_tc(const OskParams& p_in, cudaStream_t st) {
  CUtensorMap qm, km, vm;
  OskParams p = p_in;
  TileOrder vo;
  // K and V: the dense tensors, or page pools whose pages hold whole key blocks
  if (p.pg.table && p.pg.page_size < 8) return cudaErrorInvalidValue;
  const int k_box = (p.pg.table && p.pg.page_size < kBlock) ? p.pg.page_size : kBlock;   // small pages: one box per page
  const int v_box = k_box < kHalfKeys ? k_box : kHalfKeys;
  if (!make_tile_map(&qm, &p.qo, p.q, (uint64_t)p.n, (uint64_t)p.hq, (uint64_t)p.batch, p.qs) ||
      !make_kv_map(&km, &p.ko, p.k, p.pg, p.ks, p.batch, p.hkv, p.n, k_box) ||
      !make_kv_map(&vm, &vo, p.v, p.pg, p.ks, p.batch, p.hkv, p.n, v_box))
    return cudaErrorInvalidValue;
  const bool small_pages = p.pg.table && p.pg.page_size < kBlock;
  // Where the line lies, by the pitch, since the host knows no lengths.  Shared / written out, us a launch, 16K tokens of 32 heads,
  // lists of at most
  //                          4        8       16       24       32         48         64         96        128 blocks
  // Stage 2 off        112/115  179/193  316/322  446/459  562/573    811/817  1040/1038  1529/1532  2008/2010 (in one place: 107, 182, 308, 435, ...)
  // on                 111/113  167/179  277/265  362/354  425/413    554/540    693/678    917/901  1139/1116
  // on, cap half of it   95/102  128/131  209/209  304/300  393/382    540/528    665/652    918/905  1128/1101
  // (the 128K layer, Stage 2 on: 7,860/7,757; of 9 to 15 blocks 318/314, 359/350, 392/371, 420/418, 456/454, 510/500, 522/517).  With Stage 2 off the tiles' code is shared at every length, but for small pages.  Those,
  // read in place, Stage 2 off (P's first half over S and shared code, at pitches from 8 up: 8 to 12 % more than the written-out form,
  // pages of 64 2 to 4):
  //                          2        4        8       16       32         64 blocks
  // pages of 8         129/121  234/218  441/408  851/787  1663/1535  3267/3009
  // of 16              105/101  182/169  335/307  646/624  1348/1231  2575/2430
  // of 32              101/106  163/157  291/274  602/554  1173/1089  2320/2128
  // of 64              107/114  166/177  286/274  552/542  1067/1072  2118/2130
  const bool off_pages = !p.stage2 && small_pages;
  const bool long_walks = off_pages ? p.mask || p.order_stride > kShortWalkPages : p.stage2 && (p.mask || p.order_stride > kShortWalk);
  auto pick = [&](auto mask_c, auto stage2_c, auto pages_c, auto long_c) {
    return osk_tc_kernel<decltype(mask_c)::value, decltype(stage2_c)::value, decltype(pages_c)::value, decltype(long_c)::value>;
  };
  constexpr std::true_type yes{};
  constexpr std::false_type no{};
  auto kernel = off_pages ? (p.mask ? pick(yes, no, yes, yes) : (long_walks ? pick(no, no, yes, yes) : pick(no, no, yes, no)))
              : !p.stage2 ? (p.mask ? pick(yes, no, no, no) : pick(no, no, no, no))
              : p.mask    ? (small_pages ? pick(yes, yes, yes, yes) : pick(yes, yes, no, yes))
              : long_walks ? (small_pages ? pick(no, yes, yes, yes) : pick(no, yes, no, yes))
                           : (small_pages ? pick(no, yes, yes, no) : pick(no, yes, no, no));
  static SmemLimit limits[16];
  cudaError_t e = raise_smem_limit(reinterpret_cast<const void*>(kernel),
                                   &limits[(p.mask ? 8 : 0) + (p.stage2 ? 4 : 0) + (small_pages ? 2 : 0) + (long_walks ? 1 : 0)], kSmemBytes);
  if (e != cudaSuccess) return e;
  if (p.decisions) {
    size_t words = (size_t)p.batch * p.hq * p.nqb * ((p.order_stride + 31) / 32);
    e = cudaMemsetAsync(p.decisions, 0, words * 4, st);
    if (e != cudaSuccess) return e;
  }
  int32_t* status = device_status_word();
  if (!status) return cudaErrorInvalidSymbol;
  p.group = p.hq / p.hkv;
  p.by_kv = fast_div(p.group * p.nqb); p.by_group = fast_div(p.group); p.by_hkv = fast_div(p.hkv);
  const int n_sm = device_sm_count();
  p.wave = n_sm > 0 ? kCtasPerSm * n_sm : 1 << 30;   // (a CTA an item if the SM count cannot be read)
  return launch_chained(kernel, dim3(p.batch * p.hq * p.nqb), kThreads, kSmemBytes, st, qm, km, vm, p, status);
}

}  // namespace cosa
