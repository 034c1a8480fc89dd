// The per-word loop of every render: a certified FP32 filter in front of the
// exact per-word map of the render's precision.  Included at the end of
// kl_common.cuh.
#pragma once

#include "kl_common.cuh"

namespace {

// ---------------------------------------------------------------------------
// A render needs each word's pixel, not its value.  Every word's map is
// evaluated once in FP32, with a rigorous bound E on its distance from the
// value that the render's own map (FP64 or double-float) gives, and the word
// is counted into a pixel when that value cannot lie outside it.  The others
// (about 1 in 10^4: the words within E of a pixel edge) are handed to the
// exact map, 32 at a time, so the image is bit for bit the one that the exact
// map alone gives.  The FP64 pipe has 2 lanes per SM against 128 of the FP32
// pipe, and the double-float map takes 117 FP32 operations; taking them out of
// the loop is what this buys.  Near-cusp group, length 20, 8192^2: FP64
// 104.9 -> 3.3 ms, double-float 18.3 -> 3.4 ms; gasket, length 18, 4096^2:
// 11.74 -> 0.40 and 2.06 -> 0.44 ms (whole renders, the same images).
//
// Map.  With z = alpha + beta/(v + gamma), one complex scale k = 1/(sx beta)
// gives omega = k v + g, g = k gamma, and the offset from alpha in x-pixel
// units is (omega_r, omega_i) / |omega|^2; the row coordinate is in units of
// 1/kappa rows, kappa = sy/sx (rows grow downwards, which is the sign of
// omega_i).  8 packed operations and 2 reciprocal seeds per two words.
//
// Boxes.  A lane keeps a box in offset coordinates (center -ax, -ay, half
// widths hx, hy, already shrunk by E): a pixel, or a piece of the plane
// outside one window side, in either case cut to |offset| <= 8 rho, rho the
// offset of the word that opened it.  Words inside the box extend its run; an
// outside box is large, so the words outside the window (a third of the
// near-cusp group's) hardly ever end a run.  Runs that end inside cost an image
// add each: 1.09e7 adds in 7.3e7 warp steps at length 20, 8192^2, 2.8e6 in 2.7e6 at
// length 17, 4096^2, where a run end of some lane falls in nearly every step.
//
// Error bound, eps = 2^-24.  |delta omega| <= eps (11 |omega| + 8 |g|): k is
// the FP32 reciprocal of the FP32-rounded constant (6 eps, common to k v and
// g), g and v round once each, the two multiply-adds round against
// |k v| + |g|, |k v| <= |omega| + |g|.  As |offset| = 1/|omega|, a word found
// in a box with |offset| <= R has |omega| >= 1/R up to rounding, so its offset
// is off by at most 2 R eps (11 + 8 |g| R) (the factor 2 covers 1/|omega| of
// the true omega, given eps (11 + 8 |g| R) <= 1/2) plus 4 eps R for |omega|^2
// and the reciprocal seed, 3 eps R for the center and the last sum, 7 eps R
// for the box's own rounding and kappa, and the mixed map's own error against
// the same value, 19 eps R + 2 eps |g| R^2 (FP64 and double-float maps: below
// 2^-40 of that).  Sum: eps R (55 + 18 |g| R); the code takes
//   E = eps R (64 + 32 |g| R) + c0,  c0 = 4 eps (2 + 2/kappa + |axf| + |ayf|)
// (c0: the rounding of alpha's own coordinates), and certifies nothing when
// eps (64 + 32 |g| R) >= 1/4.

// ---------------------------------------------------------------------------
// exact words

// Pixel of suffix point j of letter u under prefix slot `slot` by the exact map
// of precision PREC, the arithmetic of kl_eval_words.
template <int PREC>
__device__ __forceinline__ int exact_pixel(const Tables& T, const View& V, uint32_t ns,
                                           uint32_t npairs, uint32_t slot, uint32_t u,
                                           uint32_t j) {
  const uint32_t fl = T.flags[slot];
  if (PREC == KL_DF64 && !(fl & kFallback)) {
    const DfConst K = df_const(T.predf[slot]);
    const float4* q = T.sufdf + 2ull * ((size_t)u * npairs + j / 2u);
    const float4 a = __ldg(q), b = __ldg(q + 1);
    const bool odd = j & 1u;
    const float rh = odd ? a.y : a.x, rl = odd ? a.w : a.z;
    const float ih = odd ? b.y : b.x, il = odd ? b.w : b.z;
    const DD vr = {pk(rh, rh), pk(rl, rl)}, vi = {pk(ih, ih), pk(il, il)};
    DD U, W;
    uv_df2(K, vr, vi, U, W);
    uint32_t ua, ub, va, vb;
    floor_keys(U, ua, ub);
    floor_keys(W, va, vb);
    const uint32_t col = ua - 0x4B400000u, row = va - 0x4B400000u;
    return (col < V.W && row < V.H) ? (int)(row * V.W + col) : -1;
  }
  if (PREC == KL_MIXED && (fl & kOnFp32)) {
    const Pre32 k = pre32_of(T.pre64[slot]);
    const float4 s = __ldg(T.suf32p + (size_t)u * npairs + j / 2u);
    const bool odd = j & 1u;
    float uf, vf;
    uv_pole32(k, odd ? s.y : s.x, odd ? s.w : s.z, uf, vf);
    const int col = __float_as_int(__fadd_rd(uf, 12582912.0f)) - k.kx;
    const int row = __float_as_int(__fadd_rd(vf, 12582912.0f)) - k.ky;
    return ((uint32_t)col < V.W && (uint32_t)row < V.H) ? row * (int)V.W + col : -1;
  }
  const double2 s = __ldg(T.suf64 + (size_t)u * ns + j);
  double uu, vv;
  if (fl & kDirect)
    uv_direct64(T.pre64[slot], s.x, s.y, V, uu, vv);
  else
    uv_pole64(T.pre64[slot], s.x, s.y, uu, vv);
  return pixel64(uu, vv, V);
}

// What the out-of-line exact code reads: one copy per warp or block in shared
// memory.
struct ExactCtx {
  Tables T;
  View V;
  uint32_t ns, npairs;
  uint32_t* img;
};

struct ExactTally {
  uint32_t in_window, atomics;
};

// Queue entry: prefix slot (bits 0-31), suffix letter (32-33), point (34-63).
constexpr uint32_t kPendCap = 127;
constexpr int kDone = -2;  // pixel of a lane whose remaining words are left to the exact map

// The n words of a warp's queue.  Out of line: it runs for about one word in
// 10^4 and its registers must not bind the loop.
template <int PREC>
__device__ __noinline__ ExactTally exact_queue(const ExactCtx* C, const unsigned long long* q,
                                               uint32_t n) {
  ExactTally r = {0u, 0u};
  for (uint32_t k = threadIdx.x & 31; k < n; k += 32) {
    const unsigned long long e = q[k];
    const int pix = exact_pixel<PREC>(C->T, C->V, C->ns, C->npairs, (uint32_t)e,
                                      (uint32_t)(e >> 32) & 3u, (uint32_t)(e >> 34));
    if (pix < 0) continue;
    atomicAdd(C->img + pix, 1u);
    ++r.in_window;
    ++r.atomics;
  }
  return r;
}

// Words [j0, j1) of each lane with `live` by the exact map (prefixes the filter does
// not serve: direct form, out of range; words past a full queue): the lanes'
// prefixes one after the other, split over the whole warp, or, where that takes
// about as many steps (most lanes have one, as in a view or with generators out of
// the filter's range, or there are few words), each lane its own, whose runs then
// are as long as in a render without a filter.  Near-cusp group,
// 13 letters, 900 x 800, half width 1e-14: FP64 141 -> 94 us, double-float 146 -> 98;
// 1e15, all words in one pixel: 1413 -> 269 and 1477 -> 280.
template <int PREC>
__device__ __noinline__ ExactTally exact_words(const ExactCtx* C, bool live, uint32_t slot,
                                               uint32_t u, uint32_t j0, uint32_t j1) {
  unsigned b = __ballot_sync(0xFFFFFFFFu, live);
  const uint32_t most = __reduce_max_sync(0xFFFFFFFFu, live ? j1 - j0 : 0u);
  const bool apart = 4u * __popc(b) * ((most + 31u) / 32u) >= 3u * most;
  Tally t;
  for (b = apart ? 1u : b; b; b &= b - 1u) {
    const int k = __ffs(b) - 1;
    const uint32_t first = __shfl_sync(0xFFFFFFFFu, j0, k), per = (j1 - first + 31u) / 32u;
    const uint32_t s = apart ? slot : __shfl_sync(0xFFFFFFFFu, slot, k);
    const uint32_t from = apart ? j0 : min(j1, first + (threadIdx.x & 31) * per);
    const uint32_t to = apart ? (live ? j1 : j0) : min(j1, from + per);
    for (uint32_t j = from; j < to; ++j)
      t.add(exact_pixel<PREC>(C->T, C->V, C->ns, C->npairs, s, u, j), C->img);
    // the last runs that lie in one pixel, as one add
    const unsigned has = __ballot_sync(0xFFFFFFFFu, t.run && t.cur >= 0);
    if (has) {
      const int lead = __ffs(has) - 1;
      const bool same = t.cur == __shfl_sync(0xFFFFFFFFu, t.cur, lead);
      const uint32_t mine = same ? t.run : 0u, all = __reduce_add_sync(0xFFFFFFFFu, mine);
      t.in_window += mine;
      if (same) t.run = 0;
      if ((threadIdx.x & 31) == lead) {
        atomicAdd(C->img + t.cur, all);
        ++t.atomics;
      }
    }
    t.flush(C->img);
  }
  return {t.in_window, t.atomics};
}

// ---------------------------------------------------------------------------
// the loop

// A lane's current box.
struct Box {
  f2 AX, AY;     // minus the box's center, in offset coordinates, in both halves
  float hx, hy;  // half widths less the error bound (negative: nothing certified)
};

// Opens the box of a word with offset (X, Y), whose pixel (-1: outside the
// window) goes to `pix`; true if the word itself is certified to lie in it.
__device__ __forceinline__ bool open_box(const PreF* f, const View& V, float X, float Y, Box& B,
                                         int& pix) {
  const float4 c = reinterpret_cast<const float4*>(f)[1];  // axf, ayf, eb, c0
  const int4 d = reinterpret_cast<const int4*>(f)[2];      // axi, ayi, 1/|g|, 0
  const float magic = 12582912.0f;  // 1.5 * 2^23: t bits - 0x4B400000 = floor
  const float tu = __fadd_rd(X + c.x, magic), tv = __fadd_rd((Y + c.y) * V.kappa, magic);
  // a far or non-finite word has t bits that put its column or row outside
  // the window (|axi| < 2^20, W <= 2^16)
  const int col = __float_as_int(tu) + (d.x - 0x4B400000);
  const int row = __float_as_int(tv) + (d.y - 0x4B400000);
  const float rho = fabsf(X) + fabsf(Y);
  float R = rho + (1.0f + V.ik);
  float E = fmaf(R, fmaf(c.z, R, 64.0f * kEps24), c.w);
  float cx = (tu - magic) + 0.5f - c.x, cy = fmaf((tv - magic) + 0.5f, V.ik, -c.y);
  float hx = 0.5f, hy = 0.5f * V.ik;
  const bool in = (uint32_t)col < V.W && (uint32_t)row < V.H;
  pix = in ? row * (int)V.W + col : -1;
  if (!(in && E < 0x1p-11f)) {
    // a piece of the plane outside the window, or of a pixel whose bound
    // wants smaller offsets: cut to |offset| <= lim, not below 16 c0, whose
    // share of the box would else settle nothing (a limit set in one pixel of a view
    // far out: FP64, 15 letters, 1009 -> 372 us)
    const float lim = fmaxf(8.0f * (rho + __int_as_float(d.z)), 16.0f * c.w);
    float x0 = -lim, x1 = lim, y0 = -lim, y1 = lim;
    R = 2.0f * lim;
    if (in) {
      x0 = fmaxf(x0, cx - hx);
      x1 = fminf(x1, cx + hx);
      y0 = fmaxf(y0, cy - hy);
      y1 = fminf(y1, cy + hy);
      R = fminf(R, rho + (1.0f + V.ik));
    } else {
      const float wl = (float)(-d.x) - c.x, wr = (float)((int)V.W - d.x) - c.x;
      const float wt = fmaf((float)(-d.y), V.ik, -c.y);
      const float wb = fmaf((float)((int)V.H - d.y), V.ik, -c.y);
      if (X < wl)
        x1 = fminf(x1, wl);
      else if (X > wr)
        x0 = fmaxf(x0, wr);
      else if (Y < wt)
        y1 = fminf(y1, wt);
      else
        y0 = fmaxf(y0, wb);
    }
    const float e = fmaf(c.z, R, 64.0f * kEps24);
    E = e < 0.25f ? fmaf(R, e, c.w) : __int_as_float(0x7F800000);
    cx = 0.5f * (x0 + x1);
    cy = 0.5f * (y0 + y1);
    hx = 0.5f * (x1 - x0);
    hy = 0.5f * (y1 - y0);
  }
  B.AX = pk(-cx, -cx);
  B.AY = pk(-cy, -cy);
  B.hx = hx - E;
  B.hy = hy - E;
  return fabsf(X - cx) < B.hx && fabsf(Y - cy) < B.hy;
}

// A warp's shared memory.
struct WarpQueue {
  unsigned long long e[kPendCap];  // undecided words
  uint32_t n;                      // entries (past kPendCap: not stored)
  uint32_t over[32];               // per lane: its first word that found the queue full
  unsigned long long words, fp64_words;  // of the warp's items so far
};

// One warp's share of the work on one group.  Every lane of the warp calls
// every method.
template <int PREC>
struct WordWarp {
  const ExactCtx* C;
  WarpQueue* Q;
  uint32_t in_window = 0, atomics = 0;

  __device__ __forceinline__ WordWarp(const ExactCtx* c, WarpQueue* q) : C(c), Q(q) {
    Q->n = 0;
    Q->words = Q->fp64_words = 0;
    __syncwarp();
  }

  // n words of pixel pix (-1: outside the window)
  __device__ __forceinline__ void add(int pix, uint32_t n, uint32_t* __restrict__ img) {
    if (n && pix >= 0) {
      atomicAdd(img + pix, n);
      ++atomics;
      in_window += n;
    }
  }
  // the queue's words, if there are at least `least`
  __device__ __forceinline__ void drain(uint32_t least) {
    __syncwarp();
    const uint32_t n = min(Q->n, kPendCap);
    if (n < least) return;
    const ExactTally r = exact_queue<PREC>(C, Q->e, n);
    in_window += r.in_window;
    atomics += r.atomics;
    __syncwarp();
    Q->n = 0;
    __syncwarp();
  }
  // words [j0, j1) of each lane with `live`, by the exact map
  __device__ __forceinline__ void exact(bool live, uint32_t slot, uint32_t u, uint32_t j0,
                                        uint32_t j1) {
    if (!__any_sync(0xFFFFFFFFu, live)) return;
    const ExactTally r = exact_words<PREC>(C, live, slot, u, j0, j1);
    in_window += r.in_window;
    atomics += r.atomics;
  }
  // the last words of the group, and its counts
  __device__ __forceinline__ void finish(unsigned long long* counters) {
    drain(1);
    const bool first = (threadIdx.x & 31) == 0;
    publish_counts(in_window, first ? Q->words : 0ull, first ? Q->fp64_words : 0ull, atomics,
                   counters);
    __syncwarp();
    Q->words = Q->fp64_words = 0;
    in_window = atomics = 0;
    __syncwarp();
  }

  // Words of this lane's prefix slot (live: it has one) on suffix pairs
  // [k0, k1) of letter u.
  __device__ __forceinline__ void item(const Tables& T, const View& V, uint32_t ns,
                                       uint32_t npairs, uint32_t* __restrict__ img, bool live,
                                       uint32_t slot, uint32_t u, uint32_t k0, uint32_t k1) {
    const uint32_t lane = threadIdx.x & 31, j1 = min(2u * k1, ns);
    const uint32_t fl = live ? T.flags[slot] : 0u;
    const unsigned some = __ballot_sync(0xFFFFFFFFu, live);
    const unsigned f64 = __ballot_sync(0xFFFFFFFFu, fl & kFallback);
    if (lane == 0) {
      Q->words += (unsigned long long)(j1 - 2u * k0) * __popc(some);
      if (PREC != KL_FP64) Q->fp64_words += (unsigned long long)(j1 - 2u * k0) * __popc(f64);
    }
    // prefixes without a filter, one after the other with the whole warp
    exact(fl & kNoFilter, slot, u, 2u * k0, j1);
    Q->over[lane] = j1;
    if (live && !(fl & kNoFilter)) {
      const PreF* pf = filter_slot(T, slot);
      Box B = {0, 0, -1.0f, -1.0f};
      int pix = -1;
      uint32_t run = 0, e_run = k0;  // words of the run before pair e_run; all since are in it
      const float4* src = T.suf32p + (size_t)u * npairs;
      const float4 c = *reinterpret_cast<const float4*>(pf);
      const f2 K1 = pk(c.x, c.x), K2 = pk(c.y, c.y), N2 = pk(-c.y, -c.y);
      const f2 G1 = pk(c.z, c.z), G2 = pk(c.w, c.w);
#pragma unroll 4
      for (uint32_t e = k0; e < k1; ++e) {
        const float4 s = __ldg(src + e);
        const f2 vr = pk(s.x, s.y), vi = pk(s.z, s.w);
        const f2 wr = fma2(K1, vr, fma2(N2, vi, G1));
        const f2 wi = fma2(K2, vr, fma2(K1, vi, G2));
        const f2 m = fma2(wr, wr, mul2(wi, wi));
        float ma, mb;
        upk(m, ma, mb);
        const f2 rr = pk(rcp32(ma), rcp32(mb));
        float xa, xb, ya, yb;
        upk(fma2(wr, rr, B.AX), xa, xb);
        upk(fma2(wi, rr, B.AY), ya, yb);
        if (!((fabsf(xa) < B.hx) & (fabsf(xb) < B.hx) & (fabsf(ya) < B.hy) &
              (fabsf(yb) < B.hy))) {
          // the pair left the box: its words one by one
          const f2 XX = mul2(wr, rr), YY = mul2(wi, rr);
          run += 2u * (e - e_run);
          e_run = e + 1;
#pragma unroll 1
          for (uint32_t h = 0; h < 2; ++h) {
            const uint32_t j = 2u * e + h;
            const float X = __uint_as_float((uint32_t)(h ? XX >> 32 : XX));
            const float Y = __uint_as_float((uint32_t)(h ? YY >> 32 : YY));
            if (fabsf(X + __uint_as_float((uint32_t)B.AX)) < B.hx &&
                fabsf(Y + __uint_as_float((uint32_t)B.AY)) < B.hy) {
              ++run;
            } else if (j < ns && pix != kDone) {
              // (a box may end within its pixel: the run goes on)
              const int was = pix;
              const bool sure = open_box(pf, V, X, Y, B, pix);
              if (pix != was) {
                add(was, run, img);
                run = 0u;
              }
              if (sure) {
                ++run;
              } else {
                const uint32_t k = atomicAdd(&Q->n, 1u);
                if (k < kPendCap) {
                  Q->e[k] = (unsigned long long)slot | ((unsigned long long)u << 32) |
                            ((unsigned long long)j << 34);
                } else {  // full: the rest of this lane's words by the exact map
                  Q->over[lane] = j;
                  add(pix, run, img);
                  run = 0u;
                  pix = kDone;
                  B.hx = B.hy = __int_as_float(0x7F800000);
                }
              }
            }
          }
        }
      }
      add(pix, run + 2u * (k1 - e_run), img);
    }
    __syncwarp();
    exact(Q->over[lane] < j1, slot, u, Q->over[lane], j1);
    drain(32);
  }
};

// One item: 32 prefixes of one last letter x one chunk of suffix pairs.
template <int PREC>
__device__ __forceinline__ void word_item(WordWarp<PREC>& w, uint32_t item, const Work& Wk,
                                          const Plan& L, const View& V, const Tables& T,
                                          uint32_t* __restrict__ img) {
  int x, u;
  uint32_t pb, c;
  item_of(item, Wk, x, u, pb, c);
  const uint32_t k = pb * 32 + (threadIdx.x & 31);
  const bool live = k < L.nr;
  const uint32_t slot = (uint32_t)x * L.np + L.r0 + (live ? k : 0u);
  const uint32_t k0 = c * Wk.chunk, k1 = min(L.npairs, k0 + Wk.chunk);
  w.item(T, V, L.ns, L.npairs, img, live, slot, (uint32_t)u, k0, k1);
}

}  // namespace
