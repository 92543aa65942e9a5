// Double-precision recount of a list's near ties (step 3 of the sort stage).
//
// The sort kernel leaves, in the list's row of screened scores, [0] = chained entries, [1] = kept count, then per entry
// chained_entry().  One CTA of eight warps per list: M*[r] from every row's best
// block (and the runner-up of the rows the screen could not call) and the entries' block maxima, then every entry's score
// sum_r exp(M[r,j] - M*[r]); chains are re-sorted by it, ties by ascending id, and the lists patched.  A kernel of its own
// because it wants more registers than the sort, whose lists want many CTAs: 128, two CTAs an SM (with 64 and four CTAs it spilled some
// 400 bytes: Stage 1 at 32K 166.3 us instead of 162.4, of 201 blocks with Top-p 142.4 instead of 137.8).  The products run on the FP64 matrix
// unit, eight rows by eight keys at a time: it has the vector unit's rate, but a warp issues one instruction and one read of
// the query rows per 256 products (one lane per key and eight rows: 1,024 FMAs and 512 16-byte shared-memory reads a
// block and warp, 10 k cycles; inside the sort kernel, at 40 registers, 15 to 20 k).
#pragma once

#include <math.h>

#include "common.cuh"

namespace cosa {

constexpr int kRecountThreads = 256;
constexpr int kRecountMax = 96;      // chained entries one list may have before it is left to the double-precision kernel
constexpr int kRecountRows = 64;     // sampled rows of one (possibly two-tile) query block
constexpr int kRecountQuarter = kHeadDim / 4 + 1;      // pitch of a quarter row in doubles (the quarters lie in different banks)
constexpr int kRecountPad = 4 * kRecountQuarter;       // row pitch
constexpr int kRecountChunk = 16;    // entries whose maxima are held at a time

// position in the order, tied with the next position, block id (blocks of a call: below 4096, else kap_exact.cu has no room)
__device__ __forceinline__ int chained_entry(int pos, int link, int id) { return id << 16 | 2 * pos | link; }

__device__ __forceinline__ double bf16_lo(unsigned w) { return (double)__uint_as_float(w << 16); }
__device__ __forceinline__ double bf16_hi(unsigned w) { return (double)__uint_as_float(w & 0xffff0000u); }

inline size_t kap_recount_smem_bytes(int rows, int qtiles, int nqb) {
  return (size_t)rows * qtiles * kRecountPad * 8 + (qtiles == 2 ? (size_t)nqb * 4 : 0);
}

__device__ __forceinline__ void dmma_8x8x4(double (&d)[2], double a, double b) {
  asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}

// One warp: for each of eight rows (row: this lane's, the lane / 4-th of them) the maximum over its visible sampled keys of key block
// j, in all four lanes of the row.  A lane converts the quarter of a key row that is its share of every product: the k index
// of step s is quarter * 32 + s on both sides.  key_row(c): row of the block's sampled key c.
template <typename KeyRow>
__device__ __forceinline__ double recount_rows(const KapParams& p, const double* Qs, int j, int row, int row0, int R, int lane, KeyRow key_row) {
  const int quarter = lane & 3;
  const double* q = Qs + (size_t)row * kRecountPad + quarter * kRecountQuarter;
  double best = -INFINITY;
#pragma unroll 1
  for (int c0 = 0; c0 < R; c0 += 8) {
    const uint4* key = reinterpret_cast<const uint4*>(key_row(c0 + (lane >> 2))) + quarter * 4;
    uint4 w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) w[u] = key[u];
    double d[2][2] = {{0.0, 0.0}, {0.0, 0.0}};   // two chains: even and odd steps
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const unsigned kw[4] = {w[u].x, w[u].y, w[u].z, w[u].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        dmma_8x8x4(d[0], q[u * 8 + 2 * e], bf16_lo(kw[e]));
        dmma_8x8x4(d[1], q[u * 8 + 2 * e + 1], bf16_hi(kw[e]));
      }
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {                // (column of the product: the key)
      const int kc = j * R + c0 + 2 * quarter + x;
      if (!p.causal || kc <= row0 + row) best = fmax(best, (d[0][x] + d[1][x]) * p.scale);
    }
  }
  best = fmax(best, __shfl_xor_sync(0xffffffffu, best, 1));
  return fmax(best, __shfl_xor_sync(0xffffffffu, best, 2));
}

// smem: kap_recount_smem_bytes().  All threads of a CTA of kRecountThreads call it.
__device__ __forceinline__ void kap_recount_item(const KapParams& p, const KapScreenParams& sp, int row_lo_flat, unsigned char* smem) {
  struct Tied { int pos, link; unsigned id; double s; };
  __shared__ Tied tied[kRecountMax];
  struct Best { int j, n, second; unsigned char rows[8]; };      // up to eight rows against one block: M1, or (second) M2
  __shared__ Best best[2 * kRecountRows];
  __shared__ double M1[kRecountRows], M2[kRecountRows], Mset[kRecountChunk][kRecountRows];
  __shared__ int n_best, pos_after;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int R = p.rows, T = p.qtiles, RT = R * T;
  const int i_lo = row_lo_flat % p.nqb, bh = row_lo_flat / p.nqb, h = bh % p.hq, b = bh / p.hq;
  const int i = i_lo + T - 1, g = h / (p.hq / p.hkv);
  const size_t row_lo = (size_t)row_lo_flat;
  double* Qs = reinterpret_cast<double*>(smem);
  int32_t* ids = reinterpret_cast<int32_t*>(Qs + (size_t)RT * kRecountPad);   // (T == 2) the ranking's kept ids

  const int* words = reinterpret_cast<const int*>(sp.scores + row_lo * p.nqb);
  const int nt = words[0], K = words[1];
  if (tid < nt) {
    const int w = words[2 + tid];
    tied[tid].pos = (w & 0xffff) >> 1; tied[tid].link = w & 1; tied[tid].id = (unsigned)(w >> 16);
  }
  unsigned long long amb = 0ULL;
  for (int t = 0; t < T; ++t) amb |= (unsigned long long)sp.ambmask[row_lo + t] << (t * R);
  int2 js = make_int2(0, 0);
  if (tid < RT) {
    js = reinterpret_cast<const int2*>(sp.jstar)[(size_t)bh * (p.n / p.stride) + (size_t)i_lo * R + tid];
    M1[tid] = -INFINITY; M2[tid] = -INFINITY;
  }
  if (tid == 0) n_best = 0;
  const __nv_bfloat16* qh = p.q + elem_off(p.qs, b, h, 0);
  for (int e = tid; e < RT * (kHeadDim / 8); e += kRecountThreads) {
    const int r = e / (kHeadDim / 8), c8 = e % (kHeadDim / 8);
    const uint4 w = reinterpret_cast<const uint4*>(qh + ((size_t)(i_lo * R + r) * p.stride) * p.qs.t)[c8];
    const unsigned ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int u = 0; u < 4; ++u)
      for (int x = 0; x < 2; ++x)
        Qs[(size_t)r * kRecountPad + (c8 / 4) * kRecountQuarter + (c8 % 4) * 8 + 2 * u + x] = x ? bf16_hi(ws[u]) : bf16_lo(ws[u]);
  }
  if (T == 2)
    for (int t = tid; t < K; t += kRecountThreads) ids[t] = p.order[(row_lo + 1) * p.order_stride + t];
  __syncthreads();
  // the blocks that decide M*: the rows of a warp that share their best block go together, eight at a time; the runner-ups of the
  // rows in question one by one
  if (tid < ((RT + 31) & ~31)) {
    const bool row_ok = tid < RT;
    const unsigned peers = __match_any_sync(0xffffffffu, row_ok ? js.x : -1 - lane);
    const int rank = __popc(peers & ((1u << lane) - 1u)), leader = __ffs(peers) - 1, n = __popc(peers);
    int first = 0;
    if (row_ok && rank == 0) first = atomicAdd(&n_best, (n + 7) / 8);
    first = __shfl_sync(0xffffffffu, first, leader);
    if (row_ok) {
      Best& m = best[first + rank / 8];
      m.rows[rank % 8] = (unsigned char)tid;
      if (rank % 8 == 0) { m.j = js.x; m.n = min(8, n - rank); m.second = 0; }
      if ((amb >> tid) & 1ULL) {
        Best& m2 = best[atomicAdd(&n_best, 1)];
        m2.rows[0] = (unsigned char)tid; m2.j = js.y; m2.n = 1; m2.second = 1;
      }
    }
  }
  __syncthreads();
  const int tiles = RT / 8;
  for (int base = 0; base < nt; base += kRecountChunk) {
    const int m = min(kRecountChunk, nt - base), n_first = base == 0 ? n_best : 0;
    for (int x = warp; x < n_first + m * tiles; x += kRecountThreads / 32) {
      int j, row, n = 8;
      double* out;
      if (x < n_first) {
        j = best[x].j; n = best[x].n;
        row = best[x].rows[min(lane >> 2, n - 1)];
        out = best[x].second ? M2 : M1;
      } else {
        const int y = x - n_first;
        j = (int)tied[base + y / tiles].id;
        row = (y % tiles) * 8 + (lane >> 2);
        out = Mset[y / tiles];
      }
      const double z = recount_rows(p, Qs, j, row, i_lo * R, R, lane, [&](int c) {
        return p.k + kv_off(p.pg, p.ks, b, p.hkv, g, (j * R + c) * p.stride);
      });
      if ((lane & 3) == 0 && (lane >> 2) < n) out[row] = z;
    }
    __syncthreads();
    for (int e = tid; e < m * RT; e += kRecountThreads) {
      const int x = e / RT, r = e % RT;
      Mset[x][r] = exp(Mset[x][r] - fmax(M1[r], M2[r]));   // exp(-inf) = 0: the row sees nothing of the block
    }
    __syncthreads();
    if (tid < m) {
      double sum = 0.0;
      for (int r = 0; r < RT; ++r) sum += Mset[tid][r];
      tied[base + tid].s = sum;
    }
    __syncthreads();
  }
  if (tid == 0) {
    // order the chained entries by position, then re-sort every chain by (score desc, id asc)
    for (int a = 1; a < nt; ++a) {
      Tied x = tied[a];
      int c = a - 1;
      while (c >= 0 && tied[c].pos > x.pos) { tied[c + 1] = tied[c]; --c; }
      tied[c + 1] = x;
    }
    int a = 0;
    while (a < nt) {
      int e = a;
      while (e + 1 < nt && tied[e + 1].pos == tied[e].pos + 1 && tied[e].link) ++e;
      for (int x = a + 1; x <= e; ++x) {  // insertion sort of one chain; the positions stay
        const unsigned idx = tied[x].id;
        const double sx = tied[x].s;
        int c = x - 1;
        while (c >= a && (tied[c].s < sx || (tied[c].s == sx && tied[c].id > idx))) {
          tied[c + 1].id = tied[c].id; tied[c + 1].s = tied[c].s; --c;
        }
        tied[c + 1].id = idx; tied[c + 1].s = sx;
      }
      a = e + 1;
    }
    pos_after = K;
  }
  __syncthreads();
  if (T == 1) {
    if (tid < nt && tied[tid].pos < K) p.order[row_lo * p.order_stride + tied[tid].pos] = (int32_t)tied[tid].id;
  } else {
    // both tiles' lists anew: the first leaves out the key blocks that lie wholly after it (the one block i), which a chain
    // that straddles the end of the kept prefix can move in or out
    if (tid < nt && tied[tid].pos < K) ids[tied[tid].pos] = (int32_t)tied[tid].id;
    __syncthreads();
    if (p.causal)
      for (int t = tid; t < K; t += kRecountThreads)
        if (ids[t] == i) pos_after = t;
    __syncthreads();
    for (int tile = 0; tile < T; ++tile) {
      const bool drop = tile == 0 && pos_after < K;
      const int kept = K - (drop ? 1 : 0);
      int32_t* dst = p.order + (row_lo + tile) * p.order_stride;
      for (int t = tid; t < p.order_stride; t += kRecountThreads) dst[t] = t < kept ? ids[(drop && t >= pos_after) ? t + 1 : t] : -1;
      if (tid == 0) p.count[row_lo + tile] = kept;
    }
  }
  __syncthreads();   // the shared words are the next item's
}

}  // namespace cosa
