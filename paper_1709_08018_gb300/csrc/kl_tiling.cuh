// The tiling render (every node of the word tree): all lengths that share one
// prefix table in one set of launches, and the short lengths walked as trees.
// Included by kl_render.cu.
//
// A tiling render of d letters is d renders, nearly all of them far too small
// to fill the GPU: three launches per length, each waiting for the one before,
// took 198 us for 14 letters at 1920 x 1080, whose 9.6e6 words need 10 us of
// the FP32 pipe.  The default plans of lengths 10 .. 17 split off the same nine
// prefix letters, so their words differ only in the suffix table: one parts
// launch, one combine launch and one render launch whose queue holds the items
// of all these lengths and the short lengths' nodes.  The same render: 57 to 62 us.
// Mixed lengths take the filtered loop of kl_filter.cuh here, so that one kernel
// serves the three precisions; a single mixed render keeps its own loop
// (render_mixed_kernel), whose run ends cost less (near-cusp, length 20: 2.88
// against 3.31 ms; 64 batched groups: 3.2 against 4.2 ms).
#pragma once

#include "kl_common.cuh"

namespace {

// ---------------------------------------------------------------------------
// short lengths

// Lengths 1 .. k0 <= kShortTiling: words evaluated point by point from the
// inside out (the seed of w_k, then the maps of w_k, ..., w_1), in FP64 with a
// refined reciprocal instead of division.  The point of a word is that of its
// right end (the word without w_1) under one more map, so a lane evaluates one
// word and walks the words that extend it to the left, kShortWalk letters deep:
// a fifth of the maps of evaluating every word from its seed.
constexpr uint32_t kShortTiling = 9;
constexpr int kShortWalk = 2;

// Its multiply-adds are spelled out so that a word has the same value, bit for bit,
// wherever it is evaluated (from its seed, or as a walk's first or second letter).
__device__ __forceinline__ dc short_map(const Group& G, int x, dc z) {
  return point_map(G.g + 8 * x, z);
}

// Roots of the walk: the words of lengths 1 .. short_root_length; those of the
// largest length are walked, the others stand for themselves.  Only all kShortTiling
// lengths have words enough to fill the FP64 pipe; below, the chain of one lane
// is what takes the time, and every word is a root (7 letters, 700 x 500: 23 us,
// walked 26).
__host__ __device__ __forceinline__ uint32_t short_root_length(uint32_t k0) {
  return k0 >= kShortTiling ? k0 - (uint32_t)kShortWalk : k0;
}
__host__ __device__ __forceinline__ uint32_t short_roots(uint32_t k0) {
  uint32_t total = 0, nk = 4;
  for (uint32_t k = 1; k <= short_root_length(k0); ++k, nk *= 3u) total += nk;
  return total;
}

// Root i of the lengths 1 .. k0 and its walk.
__device__ __noinline__ UnitTally short_unit(const Group* G, const View* V, uint32_t k0,
                                             uint32_t i, uint32_t* __restrict__ img) {
  UnitTally t = {0u, 0u, 0u};
  uint32_t r = i, n = 4, k = 1;
  while (r >= n) {
    r -= n;
    n *= 3u;
    ++k;
  }
  // innermost letter first: the base-3 digits of r from the right give w_k,
  // w_(k-1), ... relative to the letter before each
  int w[kShortTiling];
  decode_word(r, (int)k, w);
  const int last = w[k - 1];
  dc z = {G->seed[2 * last], G->seed[2 * last + 1]};
  for (int j = (int)k - 1; j >= 0; --j) z = short_map(*G, w[j], z);
  const uint32_t walk = k == short_root_length(k0) ? k0 - k : 0u;
  auto splat = [&](dc p) {
    const int pix = pixel64((p.re - V->x0) * V->sx, (V->y1 - p.im) * V->sy, *V);
    ++t.words;
    if (pix >= 0) {
      atomicAdd(img + pix, 1u);
      ++t.in_window;
      ++t.atomics;
    }
  };
  splat(z);
  if (walk == 0) return t;
  static_assert(kShortWalk == 2, "two levels below a root");
#pragma unroll 1
  for (int a = 0; a < 3; ++a) {
    const int x = allowed_letter(a, (w[0] + 2) & 3);
    const dc y = short_map(*G, x, z);
    splat(y);
    if (walk < 2) continue;
#pragma unroll 1
    for (int b = 0; b < 3; ++b) splat(short_map(*G, allowed_letter(b, (x + 2) & 3), y));
  }
  return t;
}

__global__ void __launch_bounds__(32) tiling_short_kernel(const __grid_constant__ Group G,
                                                          const __grid_constant__ View V,
                                                          uint32_t k0, int fp64_count,
                                                          uint32_t* __restrict__ img,
                                                          unsigned long long* counters) {
  const uint32_t total = short_roots(k0);
  uint32_t in_window = 0, words = 0, atomics = 0;
  for (uint32_t i = blockIdx.x * 32u + threadIdx.x; i < total; i += gridDim.x * 32u) {
    const UnitTally r = short_unit(&G, &V, k0, i, img);
    in_window += r.in_window;
    words += r.words;
    atomics += r.atomics;
  }
  publish_counts(in_window, words, fp64_count ? words : 0u, atomics, counters);
}

// ---------------------------------------------------------------------------
// lengths with common prefix tables

constexpr uint32_t kMaxLengths = 8;

// Longest first.  The prefix tables, and the suffix side of the longest, lie
// where the plan of the longest has them; the suffix sides of the others in
// the fallback list's place, which a filtered render does not use.
struct LengthSet {
  uint32_t n, k0;
  Plan L[kMaxLengths];
  Tables T[kMaxLengths];
  Work Wk[kMaxLengths];
  // first entry of each length in the three index spaces (parts and combine
  // after the prefix entries; items after the short lengths')
  uint32_t parts[kMaxLengths + 1], comb[kMaxLengths + 1], items[kMaxLengths + 1];
};

__host__ __device__ __forceinline__ uint32_t prefix_parts(const Plan& L) {
  return 4u * L.p3_q1 + (L.p > L.q ? 4u * L.p3_pq : 0u);
}

__device__ __forceinline__ uint32_t length_of(const uint32_t* base, uint32_t n, uint32_t idx) {
  uint32_t i = 0;
  while (i + 1 < n && base[i + 1] <= idx) ++i;
  return i;
}

__global__ void tiling_parts_kernel(Group G, const __grid_constant__ LengthSet S, int renorm,
                                    Clear C, uint32_t part_blocks, uint32_t lanes) {
  pdl_trigger();
  if (blockIdx.x < part_blocks) {
    if (blockIdx.x == 0) {
      if (threadIdx.x == 0) S.T[0].fbcount[0] = S.T[0].fbcount[1] = 0u;
      if (C.counters && threadIdx.x < KL_N_COUNTERS) C.counters[threadIdx.x] = 0ull;
    }
    const uint32_t idx = blockIdx.x * lanes + threadIdx.x;
    if (threadIdx.x < lanes && idx < S.parts[S.n]) {
      const uint32_t i = idx < S.parts[0] ? 0u : length_of(S.parts, S.n, idx);
      const uint32_t e = idx < S.parts[0] ? idx : S.parts[0] + (idx - S.parts[i]);
      part_entry(G, S.L[i], renorm, e, S.T[i]);
    }
    return;
  }
  clear_words(C.img, C.words, (size_t)(blockIdx.x - part_blocks) * blockDim.x + threadIdx.x,
              (size_t)(gridDim.x - part_blocks) * blockDim.x);
}

__global__ void tiling_combine_kernel(View V, const __grid_constant__ LengthSet S, double ptol,
                                      int prec) {
  pdl_trigger();
  pdl_wait();
  const uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < S.comb[0])
    combine_entry(V, S.L[0], ptol, prec, idx, S.T[0], 0u, nullptr, nullptr, kFilterTables);
  else if (idx < S.comb[S.n]) {
    const uint32_t i = length_of(S.comb, S.n, idx);
    suffix_entry(S.L[i], prec, idx - S.comb[i], S.T[i]);
  }
}

// Queue order: the short lengths' roots (32 to an item; long FP64 chains, so
// first), then the items of the lengths, longest first.
template <int BT, int PREC>
__global__ void __launch_bounds__(BT, 1024 / BT) tiling_words_kernel(
    const __grid_constant__ Group G, const __grid_constant__ View V,
    const __grid_constant__ LengthSet S, uint32_t* __restrict__ img,
    unsigned long long* counters) {
  __shared__ WarpQueue s_queue[BT / 32];
  __shared__ ExactCtx s_ctx[BT / 32];
  __shared__ unsigned long long s_counts[KL_N_COUNTERS];
  const uint32_t wi = threadIdx.x >> 5, lane = threadIdx.x & 31;
  ExactCtx& C = s_ctx[wi];
  block_counts_begin(s_counts);
  pdl_wait();
  WordWarp<PREC> w(&C, &s_queue[wi]);
  const uint32_t roots = short_roots(S.k0), first = S.items[0], total = S.items[S.n];
  uint32_t cur = kMaxLengths;  // the length whose context the warp holds
  for (uint32_t item = first_item_warp(); item < total;
       item = later_item_warp(S.T[0].fbcount + 1, total)) {
    if (item < first) {
      const uint32_t r = item * 32u + lane;
      UnitTally t = {0u, 0u, 0u};
      if (r < roots) t = short_unit(&G, &V, S.k0, r, img);
      w.in_window += t.in_window;
      w.atomics += t.atomics;
      const uint32_t words = __reduce_add_sync(0xFFFFFFFFu, t.words);
      if (lane == 0) {
        w.Q->words += words;
        if (PREC != KL_FP64) w.Q->fp64_words += words;
      }
      continue;
    }
    const uint32_t i = length_of(S.items, S.n, item);
    if (i != cur) {  // the undecided words are of the length before
      if (cur < kMaxLengths) w.drain(1);
      if (lane == 0) C = {S.T[i], V, S.L[i].ns, S.L[i].npairs, img};
      __syncwarp();
      cur = i;
    }
    word_item(w, item - S.items[i], S.Wk[i], S.L[i], V, C.T, img);
  }
  if (cur < kMaxLengths) w.drain(1);
  w.finish(s_counts);
  block_counts_end(s_counts, counters);
}

// ---------------------------------------------------------------------------
// host side

// Length k of a tiling render of *p: a limit-set render of the words of
// length k; the caller's prefix length applies to length d only.
inline kl_params length_params(const kl_params* p, uint32_t k) {
  kl_params q = *p;
  q.depth = k;
  q.mode = KL_LIMIT_SET;
  if (k != p->depth) q.prefix_len = 0;
  return q;
}

// The suffix side of plan L at offset `off` of the workspace; returns its end.
inline size_t place_suffix(Plan* L, bool df, size_t off) {
  const size_t nS = 4ull * L->ns;
  L->off_suf64 = off; off = align256(off + nS * sizeof(double2));
  L->off_suf32 = off; off = align256(off + 4ull * L->npairs * sizeof(float4));
  L->off_So = off; off = align256(off + 4ull * L->p3_so1 * sizeof(PartM));
  L->off_Si = off; off = align256(off + 4ull * L->p3_si1 * sizeof(double2));
  L->off_sufdf = off; off = align256(off + (df ? 8ull * L->npairs : 0) * sizeof(float4));
  return off;
}

// The lengths k, k - 1, ... > k0 that share the prefix tables of length k and
// whose suffix sides fit: S->n of them (0: length k takes a render of its own).
inline int make_lengths(const kl_params* p, uint32_t k, uint32_t k0, void* ws, int slots,
                        LengthSet* S) {
  S->n = 0;
  S->k0 = k0;
  if (p->cull) return KL_OK;
  size_t off = 0, end = 0;
  for (uint32_t j = k; j > k0 && S->n < kMaxLengths; --j) {
    const kl_params q = length_params(p, j);
    Plan& L = S->L[S->n];
    const int st = make_plan(&q, &L, false);
    if (st != KL_OK) return st;
    if (S->n == 0) {
      off = L.off_fb;
      end = L.off_fb + 4ull * L.np * sizeof(unsigned long long);
    } else {
      if (!prefix_tables_shared(S->L[0], L, p)) break;
      off = place_suffix(&L, p->precision == KL_DF64, off);
      if (off > end) break;
    }
    S->T[S->n] = carve(L, ws);
    S->Wk[S->n] = make_work(L, 32, L.npairs, slots, p->chunk_pairs);
    ++S->n;
  }
  const uint32_t pre = prefix_parts(S->L[0]);
  S->parts[0] = pre;
  S->comb[0] = 4u * S->L[0].nr;
  S->items[0] = (short_roots(k0) + 31u) / 32u;
  for (uint32_t i = 0; i < S->n; ++i) {
    S->parts[i + 1] = S->parts[i] + parts_count(S->L[i]) - pre;
    S->comb[i + 1] = S->comb[i] + 4u * S->L[i].ns;
    S->items[i + 1] = S->items[i] + S->Wk[i].n_items;
  }
  return KL_OK;
}

}  // namespace
