// General presentations: the paper's own enumeration (Sec. "Implementation")
// for any group given by an indexed Cayley table (Sec. "Cayley Multiplication
// Tables").  Every index n of the unpruned m-ary tree of depth d is d base-m
// digits plus one (symbols 1..m, w_1 most significant); the string is kept
// when the table run over it, read right to left from state 0, never reaches
// the crash state 0; a kept string is drawn at its word value (the seed of
// w_d, then the maps of w_d, ..., w_1).
//
// GPU layout.  A string is kept only if all its right ends are, and the value
// of a right end is the point that the maps further left are applied to.  So
// the kept strings are the leaves of a tree whose root side is w_d, and no
// other string is ever looked at.  Each lane takes one kept right end of d - h
// letters (a root, h <= 4), found by its rank: the numbers of kept strings of
// every length from every state, counted on the host, say which symbol the
// rank falls on.  It evaluates the root's point once and walks the root's
// subtree of h more letters depth first, one map per node.  Scanning all m^d
// strings, each kept one from its seed, took d FP64 maps per kept string and
// was bound by the FP64 pipe (2 lanes per SM).  The walk takes (d - h) / 3^h
// + 1/2 FP64 maps per kept string of the once-punctured torus: a leaf needs
// only its pixel, so its own map is made in FP32 with an error bound, and in
// FP64 (the same operations as for any node) when the bound does not settle
// the pixel (a few leaves in 100; they wait in a queue until a warp has 32).
//
// Height.  One lane walks a subtree alone, so h is the largest up to 4 that
// leaves every SM three warps of roots.  Measured at 1500 x 1100, h = 0 .. 4, torus
// table: 12 letters 386, 139, 71, 49 and 81 us (26,244 roots at h = 3, 8,748 at
// 4), 13 letters 1198, 394, 176, 112 and 96 us, 9 letters 25, 24, 26, 39 and 78;
// nine letters, every string kept: 5 letters 31, 23, 50, 305 and 2567 us, 7 letters
// 1445, 174, 123, 309 and 2644; six: 8 letters 593, 117, 82, 118 and 620.  (13 letters
// at 2000 x 1500, torus: scanning all strings took 1624 us; the FP64 pipe's
// share of the 96 is 46.)
#include "kl_common.cuh"

namespace {

constexpr int kFsaThreads = 64;
constexpr int kFsaMaxDepth = 32;
constexpr int kFsaStates = KL_FSA_MAX_LETTERS + 1;
constexpr int kFsaSubtree = 4;  // letters walked below a root, at most
constexpr uint32_t kFsaRootsPerSm = 96;

struct FsaDev {
  uint32_t m, d;
  uint8_t table[kFsaStates * kFsaStates];  // row stride m + 1
  double g[KL_FSA_MAX_LETTERS * 8];
  double seed[KL_FSA_MAX_LETTERS * 2];
  // ways[k][s]: strings of k symbols that run from state s without a crash
  unsigned long long ways[kFsaMaxDepth + 1][kFsaStates];
};

// One generator in FP32 with the 1-norms of its entries, nq and ns with kTiny
// (the leaf test).
struct FsaMap32 {
  float v[8];           // p, q, r, s (re, im)
  float np, nq, nr, ns;
};

// A block's shared tables.
struct FsaShared {
  uint32_t deg[kFsaStates];  // symbols that do not crash, per state
  uint8_t sym[kFsaStates][KL_FSA_MAX_LETTERS], to[kFsaStates][KL_FSA_MAX_LETTERS];
  double g[KL_FSA_MAX_LETTERS * 8];
  double seed[KL_FSA_MAX_LETTERS * 2];
  FsaMap32 f[KL_FSA_MAX_LETTERS];
  unsigned long long ways[kFsaMaxDepth + 1][kFsaStates];
};

// Pixel of map M of the point z (as FP32: zr, zi) where an FP32 evaluation
// settles it, -1 for certainly outside the window, kUnsettled otherwise.
// Error: numerator and denominator are sums of products of once-rounded
// values, off by at most 6 eps A and 6 eps B per part (A = |p||z| + |q|, B =
// |r||z| + |s| in 1-norms, eps = 2^-24); with 12 eps B < |den| / 4 the quotient w
// is off by less than 12 eps (A + |w| B) / |den| plus 13 eps |w| for its own
// roundings and the reciprocal root, and the pixel transform adds 5 eps of
// |w| + |x0| (|y1|); the code takes 20 eps for the last two.
// Range: a map does not change with the scale of its matrix, so entries of any
// size are legal.  |den|^2 outside (1e-30, 1e30) or |z| from 1e15 on settles
// nothing: past 1.8e19 |den|^2 overflows and the quotient and its bound would
// both be 0.  Within, what FP32 loses to underflow, 2^-150 times |z| < 2^50 in an
// entry and 2^-149 / |den|, |den| > 2^-50, in a product of the quotient, is below
// kTiny in A and B times 12 eps.
constexpr float kTiny = 0x1p-76f;
constexpr int kUnsettled = -2;
__device__ __forceinline__ int fsa_leaf32(const FsaMap32& M, float zr, float zi, const View& V,
                                          float x0, float y1, float sx, float sy) {
  const float* v = M.v;
  const float nr = fmaf(v[0], zr, fmaf(-v[1], zi, v[2])), ni = fmaf(v[0], zi, fmaf(v[1], zr, v[3]));
  const float dr = fmaf(v[4], zr, fmaf(-v[5], zi, v[6])), di = fmaf(v[4], zi, fmaf(v[5], zr, v[7]));
  const float m = fmaf(dr, dr, di * di);
  float rd;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rd) : "f"(m));
  const float rc = rd * rd;
  const float wr = fmaf(nr, dr, ni * di) * rc, wi = fmaf(ni, dr, -(nr * di)) * rc;
  const float az = fabsf(zr) + fabsf(zi), aw = fabsf(wr) + fabsf(wi);
  const float A = fmaf(M.np, az, M.nq), B = fmaf(M.nr, az, M.ns);
  const float u = (wr - x0) * sx, w = (y1 - wi) * sy;
  const float e = fmaf(12.0f * 0x1p-24f * rd, fmaf(aw, B, A), 20.0f * 0x1p-24f * aw);
  const float eu = fmaf(5.0f * 0x1p-24f, fabsf(x0), e) * sx;
  const float ew = fmaf(5.0f * 0x1p-24f, fabsf(y1), e) * sy;
  if (!(m > 1e-30f && m < 1e30f && az < 1e15f && 12.0f * 0x1p-24f * B * rd < 0.25f &&
        eu < 0.25f && ew < 0.25f))
    return kUnsettled;
  const float W = (float)V.W, H = (float)V.H;
  if (u < -eu || u > W + eu || w < -ew || w > H + ew) return -1;
  const int c0 = (int)floorf(u - eu), c1 = (int)floorf(u + eu);
  const int r0 = (int)floorf(w - ew), r1 = (int)floorf(w + ew);
  if (c0 != c1 || r0 != r1 || c0 < 0 || r0 < 0 || c0 >= (int)V.W || r0 >= (int)V.H)
    return kUnsettled;
  return r0 * (int)V.W + c0;
}

// A warp's queue of leaves that FP32 did not settle: the parent's point and
// the generator.
struct FsaQueue {
  double zr[64], zi[64];
  uint32_t x[64];
};

// What a walk carries along.  All lanes of a warp walk together (`on`: this
// lane's node exists), over the largest number of symbols any state has.
struct FsaWalk {
  const FsaShared* S;
  FsaQueue* Q;
  View V;
  float x0, y1, sx, sy;
  uint32_t* img;
  uint32_t most, len, words;
  Tally t;
};

__device__ __forceinline__ void fsa_word(FsaWalk& w, dc z) {
  w.t.add(pixel64((z.re - w.V.x0) * w.V.sx, (w.V.y1 - z.im) * w.V.sy, w.V), w.img);
}
// queue entries [len - n, len), one per lane
__device__ __forceinline__ void fsa_drain(FsaWalk& w, uint32_t n) {
  __syncwarp();
  const uint32_t lane = threadIdx.x & 31, k = w.len - n + lane;
  if (lane < n) fsa_word(w, point_map(w.S->g + 8 * w.Q->x[k], {w.Q->zr[k], w.Q->zi[k]}));
  w.len -= n;
  __syncwarp();
}

// The kept strings h letters further left of a right end with point z that
// left the run in `state`.
template <int h>
__device__ __forceinline__ void fsa_walk(FsaWalk& w, bool on, uint32_t state, dc z) {
  const FsaShared& S = *w.S;
  if constexpr (h == 0) {
    if (on) fsa_word(w, z);
    w.words += on;
  } else if constexpr (h == 1) {
    const uint32_t n = on ? S.deg[state] : 0u;
    const float zr = f32_of(z.re), zi = f32_of(z.im);
    w.words += n;
#pragma unroll 1
    for (uint32_t k = 0; k < w.most; ++k) {
      int pix = -1;
      uint32_t x = 0;
      if (k < n) {
        x = S.sym[state][k];
        pix = fsa_leaf32(S.f[x], zr, zi, w.V, w.x0, w.y1, w.sx, w.sy);
        if (pix != kUnsettled) w.t.add(pix, w.img);
      }
      const unsigned b = __ballot_sync(0xFFFFFFFFu, pix == kUnsettled);
      if (b) {
        if (pix == kUnsettled) {
          const uint32_t at = w.len + __popc(b & ((1u << (threadIdx.x & 31)) - 1u));
          w.Q->zr[at] = z.re;
          w.Q->zi[at] = z.im;
          w.Q->x[at] = x;
        }
        w.len += __popc(b);
        if (w.len >= 32) fsa_drain(w, 32);
      }
    }
  } else {
    const uint32_t n = on ? S.deg[state] : 0u;
#pragma unroll 1
    for (uint32_t k = 0; k < w.most; ++k) {
      const bool child = k < n;
      const uint32_t x = child ? S.sym[state][k] : 0u;
      fsa_walk<h - 1>(w, child, child ? S.to[state][k] : 0u, point_map(S.g + 8 * x, z));
    }
  }
}

template <int h>
__global__ void __launch_bounds__(kFsaThreads) fsa_render_kernel(
    const __grid_constant__ FsaDev F, View V, uint32_t* __restrict__ img,
    unsigned long long* counters) {
  __shared__ FsaShared S;
  __shared__ FsaQueue queues[kFsaThreads / 32];
  const uint32_t m = F.m;
  for (uint32_t i = threadIdx.x; i < 8u * m; i += kFsaThreads) S.g[i] = F.g[i];
  for (uint32_t i = threadIdx.x; i < 2u * m; i += kFsaThreads) S.seed[i] = F.seed[i];
  for (uint32_t i = threadIdx.x; i < 8u * m; i += kFsaThreads) S.f[i / 8].v[i % 8] = (float)F.g[i];
  for (uint32_t i = threadIdx.x; i < (F.d + 1) * kFsaStates; i += kFsaThreads)
    S.ways[i / kFsaStates][i % kFsaStates] = F.ways[i / kFsaStates][i % kFsaStates];
  if (threadIdx.x <= m) {
    const uint32_t s = threadIdx.x;
    uint32_t n = 0;
    for (uint32_t y = 1; y <= m; ++y) {
      const uint32_t to = F.table[s * (m + 1) + y];
      if (!to) continue;
      S.sym[s][n] = (uint8_t)(y - 1);
      S.to[s][n++] = (uint8_t)to;
    }
    S.deg[s] = n;
  }
  __syncthreads();
  if (threadIdx.x < m) {
    FsaMap32& f = S.f[threadIdx.x];
    f.np = fabsf(f.v[0]) + fabsf(f.v[1]);
    f.nq = fabsf(f.v[2]) + fabsf(f.v[3]) + kTiny;
    f.nr = fabsf(f.v[4]) + fabsf(f.v[5]);
    f.ns = fabsf(f.v[6]) + fabsf(f.v[7]) + kTiny;
  }
  __syncthreads();
  FsaWalk w = {&S, &queues[threadIdx.x / 32], V, (float)V.x0, (float)V.y1, (float)V.sx,
               (float)V.sy, img, 0u, 0u, 0u, Tally()};
  for (uint32_t s = 1; s <= m; ++s) w.most = max(w.most, S.deg[s]);  // (0 only starts a run)
  const uint32_t l = F.d - h;
  const unsigned long long roots = F.ways[l][0];
  for (unsigned long long first = blockIdx.x * (unsigned long long)kFsaThreads;
       first < roots; first += (unsigned long long)gridDim.x * kFsaThreads) {
    const bool on = first + threadIdx.x < roots;
    // the root of that rank, innermost letter first
    unsigned long long r = on ? first + threadIdx.x : 0ull;
    uint32_t state = 0;
    dc z = {0.0, 0.0};
#pragma unroll 1
    for (uint32_t k = 0; k < l; ++k) {
      uint32_t i = 0;
      for (;; ++i) {
        const unsigned long long c = S.ways[l - 1 - k][S.to[state][i]];
        if (r < c) break;
        r -= c;
      }
      const uint32_t x = S.sym[state][i];
      state = S.to[state][i];
      if (k == 0) z = {S.seed[2 * x], S.seed[2 * x + 1]};
      z = point_map(S.g + 8 * x, z);
    }
    fsa_walk<h>(w, on, state, z);
  }
  fsa_drain(w, w.len);
  w.t.flush(img);
  publish_counts(w.t.in_window, w.words, w.words, w.t.atomics, counters);
}

using FsaKernel = void (*)(FsaDev, View, uint32_t*, unsigned long long*);

int fsa_check(const kl_fsa* f, uint32_t d) {
  if (!f || f->m < 1 || f->m > KL_FSA_MAX_LETTERS) return KL_EINVAL;
  if (d < 1 || d > (uint32_t)kFsaMaxDepth) return KL_ERANGE;
  const uint32_t m = f->m;
  for (uint32_t i = 0; i < (m + 1) * (m + 1); ++i)
    if (f->table[(i / (m + 1)) * (KL_FSA_MAX_LETTERS + 1) + i % (m + 1)] > m) return KL_EINVAL;
  for (uint32_t k = 0; k < 8 * m; ++k)
    if (!isfinite(f->gens[k])) return KL_EINVAL;
  for (uint32_t k = 0; k < 2 * m; ++k)
    if (!isfinite(f->seeds[k])) return KL_EINVAL;
  unsigned long long n = 1;
  for (uint32_t k = 0; k < d; ++k) {
    if (n > (1ull << 40) / m) return KL_ERANGE;
    n *= m;
  }
  return KL_OK;
}

// ways[k][s] of FsaDev for k <= depth.
void fsa_ways(const kl_fsa* f, uint32_t depth,
              unsigned long long (*ways)[kFsaStates]) {
  const uint32_t m = f->m;
  for (uint32_t s = 0; s <= m; ++s) ways[0][s] = 1;
  // one more symbol in front: the sum over symbols of the non-crash targets' ways
  for (uint32_t k = 0; k < depth; ++k)
    for (uint32_t s = 0; s <= m; ++s) {
      unsigned long long acc = 0;
      for (uint32_t sym = 1; sym <= m; ++sym) {
        const uint32_t to = f->table[s * kFsaStates + sym];
        if (to != 0) acc += ways[k][to];
      }
      ways[k + 1][s] = acc;
    }
}

}  // namespace

extern "C" int kl_fsa_count(const kl_fsa* f, uint32_t depth, uint64_t* count) {
  const int st = fsa_check(f, depth);
  if (st != KL_OK) return st;
  if (!count) return KL_EINVAL;
  unsigned long long ways[kFsaMaxDepth + 1][kFsaStates];
  fsa_ways(f, depth, ways);
  *count = ways[depth][0];
  return KL_OK;
}

extern "C" int kl_render_fsa(const kl_fsa* f, const kl_params* p, uint32_t* d_image,
                             uint64_t* d_counters, void* d_workspace, size_t workspace_bytes,
                             void* stream) {
  if (!p || !d_image || !valid_view(p)) return KL_EINVAL;
  if (p->precision != KL_FP64) return KL_EINVAL;
  const int st = fsa_check(f, p->depth);
  if (st != KL_OK) return st;
  if (!d_workspace || ((uintptr_t)d_workspace & 255u) != 0) return KL_EINVAL;
  if (workspace_bytes < KL_FSA_WORKSPACE_BYTES) return KL_ENOSPACE;
  cudaStream_t s = (cudaStream_t)stream;
  unsigned long long* cnt = (unsigned long long*)d_counters;
  if (!p->accumulate) {
    if (cudaMemsetAsync(d_image, 0, (size_t)p->width * p->height * sizeof(uint32_t), s) !=
        cudaSuccess)
      return KL_ECUDA;
    if (cnt && cudaMemsetAsync(cnt, 0, KL_N_COUNTERS * sizeof(uint64_t), s) != cudaSuccess)
      return KL_ECUDA;
  }
  FsaDev F;
  F.m = f->m;
  F.d = p->depth;
  for (uint32_t i = 0; i < (F.m + 1) * (F.m + 1); ++i)
    F.table[i] = f->table[(i / (F.m + 1)) * (KL_FSA_MAX_LETTERS + 1) + i % (F.m + 1)];
  for (uint32_t k = 0; k < 8 * F.m; ++k) F.g[k] = f->gens[k];
  for (uint32_t k = 0; k < 2 * F.m; ++k) F.seed[k] = f->seeds[k];
  fsa_ways(f, F.d, F.ways);
  int sms = 0, occ = 0;
  if ((sms = sm_count()) <= 0) return KL_ECUDA;
  uint32_t h = F.d - 1 < (uint32_t)kFsaSubtree ? F.d - 1 : (uint32_t)kFsaSubtree;
  while (h > 0 && F.ways[F.d - h][0] < kFsaRootsPerSm * (unsigned long long)sms) --h;
  const FsaKernel kernels[kFsaSubtree + 1] = {fsa_render_kernel<0>, fsa_render_kernel<1>,
                                              fsa_render_kernel<2>, fsa_render_kernel<3>,
                                              fsa_render_kernel<4>};
  if (device_slots((const void*)kernels[h], kFsaThreads, &sms, &occ) != KL_OK) return KL_ECUDA;
  const unsigned long long roots = F.ways[F.d - h][0];
  const unsigned long long blocks = (roots + kFsaThreads - 1) / kFsaThreads;
  const unsigned long long most = (unsigned long long)sms * occ;
  if (blocks == 0) return KL_OK;
  kernels[h]<<<(unsigned)(blocks < most ? blocks : most), kFsaThreads, 0, s>>>(F, make_view(p),
                                                                            d_image, cnt);
  return check_launch();
}
