// NL-means-regularised segmentation, the second comparison model of Sec. 4:
// the gradient of the TV model replaced by a matrix D built from patch
// similarities of the image f.
//
// Graph (once per image): the patch distance d_a(i, j) = sum over the p x p
// patch of G_a(t) sum_ch (f(i + t) - f(j + t))^2 (G_a the Gaussian of
// standard deviation a normalised to sum 1, f mirrored at the border) for
// every candidate j of the varpi x varpi search window (clipped to the image)
// is computed on the GPU (in FP32, and in FP64 with every product and sum
// rounded separately where that decides the order), and each pixel's
// candidates are ranked by (distance, raster index).  The selection is sequential in the paper (pixels in
// raster order pick min(mt, 2 mt - l) new neighbours, l the neighbours they
// already have, and links are symmetric); a candidate already linked or holding
// 2 mt neighbours is passed over.  Pixels whose windows are apart don't see one
// another, so it runs as a wavefront over the image with the same result.
//
// ADMM (Sec. 3 with S replaced by D, per iteration):
//   u   = (I + D^T D)^(-1) [ D^T (v - b_v) + (w - b_w) - gamma s ]
//   v   = group shrinkage of g = b_v + D u over the m K values of a pixel,
//         b_v = g - v (kept as b_v and d = v - b_v)
//   w   = simplex projection of b_w + u, b_w = b_w + u - w.
// D^T D = 2 L (L the graph Laplacian of the symmetric neighbour sets), so
// I + D^T D has its spectrum in [1, 1 + 4 deg_max]; the u-step runs a fixed
// number of Chebyshev iterations on that interval from the previous u (no
// inner products, one launch per step), enough for a relative error below
// 1e-7 of the initial one.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "shearseg.h"
#include "shf_fast.h"
#include "shf_internal.h"
#include "shf_simplex.cuh"

struct nl_state {
  int H = 0, W = 0, K = 0, C = 0, m = 0, device = 0, deg_max = 0;
  float gamma = 1.f, lambda = 0.f;
  nl_params prm{};
  std::vector<float> codebook;
  // pinned: the links as window codes [P][kMaxM] in the order of selection, their counts
  unsigned char *codes_host = nullptr, *deg_host = nullptr;
  std::vector<float> cheb_a, cheb_c;    // Chebyshev coefficients per step
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  float *f = nullptr, *s = nullptr, *u = nullptr, *w = nullptr, *bw = nullptr, *gap = nullptr;
  // four labels per float4, Q = ceil(K/4), labels past K zero: pixel-major
  // ([P][Q]) the u-step's vectors (two Chebyshev iterates, the Chebyshev
  // direction, the right-hand side) and q = (w - b_w) - gamma s; [Q][m][P] the
  // pair b_v and d = v - b_v of the differences to the m neighbours
  float4 *xa = nullptr, *xb = nullptr, *cd = nullptr, *rhs = nullptr, *q = nullptr, *bv = nullptr, *d = nullptr;
  int Q = 0;
  int* nbr = nullptr;                   // [m][P]
  short* off = nullptr;                 // [m][P] neighbour minus pixel index (|off| <= 7 W + 7)
  unsigned char *rev = nullptr, *deg = nullptr;
  // the graph's construction: patch weights, the ranks of rank_rows rows, the selected links
  double* gw = nullptr;
  unsigned char* rank = nullptr;
  int rank_rows = 0;
  uint4* codes = nullptr;
  int* labels = nullptr;
  int* flag = nullptr;
  double* red = nullptr;
  // the persistent Chebyshev solve (K <= 4 and the image within one resident
  // grid): its barrier counter and timeout flag, the steps' (a, c), its grid
  unsigned* cbar = nullptr;
  int* cerr = nullptr;
  float2* cheb_ac = nullptr;
  int cheb_grid = 0, cheb_halo = 0;
  int iter = 0;
  cudaGraphExec_t exec = nullptr;
  bool graph_tried = false;
  size_t P() const { return static_cast<size_t>(H) * W; }
};

namespace {

constexpr int kThreads = 256;
constexpr int kRedBlocks = 512;
constexpr int kMaxM = 16;       // neighbours per pixel (2 mt, mt <= 8)
constexpr int kMaxWin = 15;     // search window side: (2r + 1)^2 <= 225 window codes
constexpr int kMaxPatch = 9;    // patch side
constexpr int kRankWarps = 8;   // warps per CTA of the ranking kernel

__device__ __forceinline__ int mirror_idx(int x, int n) {
  while (x < 0 || x >= n) x = x < 0 ? -x : 2 * (n - 1) - x;
  return x;
}

// Ranks of the window candidates of every pixel by (distance, code), code c =
// (dy + r)(2r + 1) + (dx + r) (the centre and codes outside the image
// excluded): codes in increasing order are candidates in increasing raster
// index, so this is the order (distance, raster index) of the FP64 distances
// with every product and sum rounded separately.
//
// GB300's FP64 rate is a 64th of its FP32 rate, and the exact distances are
// only needed where they decide the order.  A warp takes a pixel: FP32
// distances from a shared-memory tile of the image (7 candidates per lane),
// a bitonic sort of (distance, code) keys over the warp's registers, and then,
// for the candidates whose FP32 distance is within twice its error bound of a
// neighbour's in the sorted order, the FP64 distances, by which each run of
// such candidates is ordered.  The bound: with the weights and the image
// in the range checked below, a distance is a sum of n positive terms, each
// with four rounding errors, so its relative error is at most (n + 4) 2^-24
// (the caller's `delta` doubles it) plus what underflow costs (kTiny).  Rounding
// the bound itself costs nothing: a distance above the rounded bound is at least
// the next number up, which lies above the exact one.
constexpr int kRankTX = 32, kRankTY = 4;  // pixels per CTA
constexpr int kMaxHalo = kMaxWin / 2 + kMaxPatch / 2;
constexpr int kRankRows = kRankTY + 2 * kMaxHalo, kRankCols = kRankTX + 2 * kMaxHalo;
constexpr float kRankMax = 1e4f;  // largest |f| of a tile for the FP32 distances
constexpr float kTiny = 1e-36f;
// ranks of a pixel, padded to whole words, and the bytes of them held at a time
// (512 x 512 takes 67 MB, in one go)
constexpr int kRankPitch = 256;
constexpr size_t kRankBytes = size_t{256} << 20;
constexpr size_t kRingBytes = 200 * 1024;  // shared memory for the selection's counts

// FP64 distance of the pixel at tile position (y, x) to the candidate (dy, dx).
__device__ __forceinline__ double nl_exact(const float (*tile)[kRankRows][kRankCols], int C, const double* __restrict__ G,
                                           int h, int y, int x, int dy, int dx) {
  const int n = 2 * h + 1;
  double acc = 0.0;
  for (int t1 = -h; t1 <= h; ++t1)
    for (int t2 = -h; t2 <= h; ++t2) {
      double sum = 0.0;
      for (int ch = 0; ch < C; ++ch) {
        const double dd = __dsub_rn(static_cast<double>(tile[ch][y + t1][x + t2]),
                                    static_cast<double>(tile[ch][y + dy + t1][x + dx + t2]));
        sum = __dadd_rn(sum, __dmul_rn(dd, dd));
      }
      acc = __dadd_rn(acc, __dmul_rn(G[(t1 + h) * n + (t2 + h)], sum));
    }
  return acc;
}

// The rows from ystrip up to yend.  rank [pixels][kRankPitch] holds every code of
// those rows' pixels in order, 255 for the unused positions at the end; word w of
// the pixel's 64 holds the positions 64 (w / 16) + w % 16 + {0, 16, 32, 48}.  G: the patch weights [(2h+1)^2].
// Bound by instruction issue (about 3000 warp instructions a pixel: distances
// 900, sort 1500); 512 x 512, 5 x 5 patches, 15 x 15 window: 79.3 ms with FP64
// distances and ranks counted over all pairs, 1.2 ms so.
template <int C>
__global__ void __launch_bounds__(32 * kRankWarps)
    k_nl_rank(const float* __restrict__ f, int H, int W, const double* __restrict__ G, int h, int r, float delta,
              int ystrip, int yend, unsigned char* __restrict__ rank) {
  __shared__ float tile[C][kRankRows][kRankCols];
  __shared__ float sG[kMaxPatch * kMaxPatch];
  __shared__ double ex[kRankWarps][256];
  __shared__ __align__(8) unsigned char out[kRankWarps][kRankPitch];
  __shared__ unsigned char code[kRankWarps][256], list[kRankWarps][256], near_next[kRankWarps][256];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int side = 2 * r + 1, NW = side * side, cen = NW / 2, n = 2 * h + 1, halo = r + h;
  const size_t P = static_cast<size_t>(H) * W;
  const int y0 = ystrip + blockIdx.y * kRankTY, x0 = blockIdx.x * kRankTX;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) sG[e] = static_cast<float>(G[e]);
  // the image around the CTA's pixels, mirrored at the borders
  const int rows = kRankTY + 2 * halo, cols = kRankTX + 2 * halo;
  bool wide = false;
  for (int e = threadIdx.x; e < rows * cols; e += blockDim.x) {
    const int y = e / cols, x = e - y * cols;
    const size_t src = static_cast<size_t>(mirror_idx(y0 - halo + y, H)) * W + mirror_idx(x0 - halo + x, W);
#pragma unroll
    for (int ch = 0; ch < C; ++ch) {
      const float v = f[ch * P + src];
      tile[ch][y][x] = v;
      wide = wide || !(fabsf(v) <= kRankMax);
    }
  }
  // delta < 0: weights too small for the bound; then, and for large values,
  // every candidate takes its FP64 distance
  const bool all_exact = __syncthreads_or(wide ? 1 : 0) != 0 || delta < 0.f;
  // the lane's candidates: number lane + 32 q of the window without its centre
  int dy[7], dx[7];
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    const int m = lane + 32 * q, c = m < cen ? m : m + 1;
    dy[q] = m < NW - 1 ? c / side - r : 0;
    dx[q] = m < NW - 1 ? c % side - r : 0;
  }
  for (int px = wid; px < kRankTX * kRankTY; px += kRankWarps) {
    const int ri = y0 + px / kRankTX, ci = x0 + px % kRankTX;
    if (ri >= yend || ci >= W) continue;  // the whole warp
    const int y = px / kRankTX + halo, x = px % kRankTX + halo;
    float acc[7];
    const float* base[7];
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      acc[q] = 0.f;
      base[q] = &tile[0][y + dy[q] - h][x + dx[q] - h];
    }
    const float* own = &tile[0][y - h][x - h];
#pragma unroll
    for (int ch = 0; ch < C; ++ch)
      for (int t1 = 0; t1 < n; ++t1)
        for (int t2 = 0; t2 < n; ++t2) {
          const int o = (ch * kRankRows + t1) * kRankCols + t2;
          const float a = own[o], g = sG[t1 * n + t2];
#pragma unroll
          for (int q = 0; q < 7; ++q) {
            const float d = a - base[q][o];
            acc[q] = fmaf(d * g, d, acc[q]);
          }
        }
    // keys: distance bits (non-negative floats order as integers) and code
    unsigned long long key[8];
    int nv = 0;  // valid candidates
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      const int m = lane + 32 * q, c = m < cen ? m : m + 1;
      const int rj = ri + dy[q], cj = ci + dx[q];
      const bool ok = m < NW - 1 && rj >= 0 && rj < H && cj >= 0 && cj < W;
      const unsigned bits = all_exact ? 0u : __float_as_uint(acc[q]);
      key[q] = ok ? (static_cast<unsigned long long>(bits) << 32) | static_cast<unsigned>(c) : ~0ull;
      nv += __popc(__ballot_sync(0xffffffffu, ok));
    }
    key[7] = ~0ull;
    // bitonic sort of the 256 keys, element lane * 8 + i in key[i]
#pragma unroll
    for (int k = 2; k <= 256; k <<= 1)
#pragma unroll
      for (int j = k >> 1; j > 0; j >>= 1) {
        if (j >= 8) {
          const bool up = ((lane * 8) & k) == 0, lower = (lane & (j / 8)) == 0;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, key[i], j / 8);
            key[i] = ((o < key[i]) == (up == lower)) ? o : key[i];
          }
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if ((i & j) == 0) {
              const bool up = ((lane * 8 + i) & k) == 0;
              const unsigned long long a = key[i], b = key[i | j];
              const bool sw = (b < a) == up;
              key[i] = sw ? b : a;
              key[i | j] = sw ? a : b;
            }
        }
      }
    // which neighbours in the order are closer than the bound
    const unsigned long long first_next = __shfl_down_sync(0xffffffffu, key[0], 1);
    unsigned close = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int e = lane * 8 + i;
      const float a = __uint_as_float(static_cast<unsigned>(key[i] >> 32));
      const float b = __uint_as_float(static_cast<unsigned>((i < 7 ? key[i < 7 ? i + 1 : 0] : first_next) >> 32));
      const bool c = e + 1 < nv && !(b > fmaf(a, delta, a) + kTiny);
      close |= (c ? 1u : 0u) << i;
      code[wid][e] = static_cast<unsigned char>(key[i]);
      out[wid][e] = e < nv ? static_cast<unsigned char>(key[i]) : 255;
      near_next[wid][e] = c ? 1 : 0;
    }
    const unsigned before = __shfl_up_sync(0xffffffffu, close, 1) >> 7;
    const unsigned amb = close | ((close << 1) & 0xffu) | (lane > 0 ? before & 1u : 0u);
    if (__any_sync(0xffffffffu, amb != 0u)) {
      // positions of the undecided candidates
      int at = __popc(amb), total = at;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, at, o);
        at += lane >= o ? v : 0;
      }
      total = __shfl_sync(0xffffffffu, at, 31);
      at -= __popc(amb);
      for (int i = 0; i < 8; ++i)
        if (amb >> i & 1u) list[wid][at++] = static_cast<unsigned char>(lane * 8 + i);
      __syncwarp();
      for (int q = lane; q < total; q += 32) {
        const int e = list[wid][q], c = code[wid][e];
        ex[wid][e] = nl_exact(tile, C, G, h, y, x, c / side - r, c % side - r);
      }
      __syncwarp();
      for (int q = lane; q < total; q += 32) {
        const int e = list[wid][q];
        const double me = ex[wid][e];
        const int c = code[wid][e];
        int pos = e;
        for (int o = e - 1; o >= 0 && near_next[wid][o]; --o) {
          const double v = ex[wid][o];
          pos -= (v > me || (v == me && code[wid][o] > c)) ? 1 : 0;
        }
        for (int o = e + 1; near_next[wid][o - 1]; ++o) {
          const double v = ex[wid][o];
          pos += (v < me || (v == me && code[wid][o] < c)) ? 1 : 0;
        }
        out[wid][pos] = static_cast<unsigned char>(c);
      }
    }
    __syncwarp();
    const size_t i = static_cast<size_t>(ri) * W + ci;
    unsigned word[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int w = 2 * lane + q;
      const unsigned char* o = out[wid] + (w & ~15) * 4 + (w & 15);
      word[q] = o[0] | static_cast<unsigned>(o[16]) << 8 | static_cast<unsigned>(o[32]) << 16 |
                static_cast<unsigned>(o[48]) << 24;
    }
    reinterpret_cast<uint2*>(rank + (i - static_cast<size_t>(ystrip) * W) * kRankPitch)[lane] = make_uint2(word[0], word[1]);
    __syncwarp();
  }
}

// The selection for the rows [y0, y0 + rows), whose ranks are in `rank`, after
// every row above: codes [P][kMaxM] holds the window codes of a pixel's links in the
// order they were made (255 for none), deg [P] their number.
//
// A pixel reads and changes the state of its window only, and two pixels can
// meet in a window only if their columns are at most 2 r apart.  So at step t one
// CTA takes the pixel (y, t - S y) of every row y, S = 2 r + 1: pixels of one step
// have disjoint windows, and of any two pixels that meet the earlier one in
// raster order comes in an earlier step (its row is d rows up, its column at
// most 2 r < S d further right).  The links, their order included, are those of
// the raster loop.  A half warp takes a pixel, 16 candidates at a time in the
// order of rank; with more rows than half warps a step takes several turns.
//
// Bound by one SM's latency and issue slots, W + S (rows - 1) steps of two
// dependent shared-memory reads, the votes and a barrier.  Hence
//  - RING: the counts of the rows in reach live in shared memory, row y in slot
//    y mod R; a row enters with the first row that reaches it, when the row R above,
//    which no pixel reaches any more, goes to memory (R >= 2 r + (W - 1) / S + 1).
//    Otherwise (images too wide for that) the counts are read from L2.
//  - the next pixel's first 64 candidates and own links are read a step ahead; of the
//    pixels that can link to it in between, there is only the current one.
// A step takes about 1.1 us (512 x 512, window 15: 8177 steps, 9 ms).  The graph of an
// image, with the raster loop on the host and the copies of ranks and links, and so:
// 256 x 256 4.5 and 4.5 ms, 512 x 512 17.6 and 11.2, 1024 x 1024 68 and 42, 1800 x
// 1800 212 and 105, 2048 x 2048 (counts in L2) 274 and 146; a 64 x 64 image, 0.56 and
// 1.13, is the price of one path.  64 candidates at a time (four per lane) took 25 ms
// at 512 x 512: the step is bound by instructions as much as by its chain.
template <bool RING>
__global__ void __launch_bounds__(1024) k_nl_select(const unsigned* __restrict__ rank, int H, int W, int r, int m,
                                                    int mt, int y0, int rows, int R, unsigned char* codes,
                                                    unsigned char* deg) {
  __shared__ int step[256];
  extern __shared__ unsigned char ring[];
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int kWords = kRankPitch / 4;
  const int side = 2 * r + 1, NW = side * side;
  const int lane = threadIdx.x & 31, gl = lane & 15, grp = threadIdx.x >> 4, ngrp = blockDim.x >> 4;
  const int turns = (min(rows, (W + side - 1) / side) + ngrp - 1) / ngrp, slots = turns * ngrp;
  const int right = NW / 2 + 1, left_code = NW / 2 - 1;  // the codes of the row's next and previous pixel
  for (int c = threadIdx.x; c < NW; c += blockDim.x) step[c] = (c / side - r) * W + (c % side - r);
  const int first = max(0, y0 - r), RW = R * W;
  if (RING)
    for (int y = first; y < min(H, y0 + r); ++y)
      for (int x = threadIdx.x; x < W; x += blockDim.x) ring[(y % R) * W + x] = deg[y * W + x];
  __syncthreads();
  unsigned char* const count = RING ? ring : deg;
  const int steps = W + side * (rows - 1);
  int yn = -1, xn = 0;  // the pixel that was read ahead: candidates, own links, linked by the one before
  unsigned cn = kAll;
  uint4 on = make_uint4(0u, 0u, 0u, 0u);
  bool ln = false;
  // the rows [ylo, yhi] of the step; ymod = ylo mod slots
  int ylo = 0, yhi = -1, ymod = 0, start = 0, end = W;
  for (int t = 0; t < steps; ++t) {
    if (t == end) {  // the first row is done
      ++ylo;
      end += side;
      ymod = ymod + 1 == slots ? 0 : ymod + 1;
    }
    if (t == start && yhi + 1 < rows) {  // a row starts
      ++yhi;
      start += side;
      const int e = y0 + yhi + r;
      if (RING && e < H) {  // row e enters
        for (int x = threadIdx.x; x < W; x += blockDim.x) {
          unsigned char* at = ring + (e % R) * W + x;
          if (e - R >= first) deg[(e - R) * W + x] = *at;
          *at = 0;
        }
        __syncthreads();
      }
    }
    for (int turn = 0; turn < turns; ++turn) {
      const int slot = turn * ngrp + grp;
      const int y = ylo + slot - ymod + (slot < ymod ? slots : 0), x = t - side * y;
      const bool act = y <= yhi;
      const int i = act ? (y0 + y) * W + x : 0;                       // the pixel
      const int ci = RING ? (act ? ((y0 + y) % R) * W + x : 0) : i;   // where its count is
      const unsigned* rk = rank + (act ? static_cast<size_t>(y * W + x) * kWords : 0) + gl;
      int left = 0, dgi = 0;
      unsigned cw = kAll;  // the lane's next four candidates, 255 for none
      uint4 own = make_uint4(0u, 0u, 0u, 0u);
      bool link_left = false;
      if (act) {
        dgi = count[ci];
        left = min(mt, m - dgi);
        if (y == yn && x == xn) {
          cw = cn;
          own = on;
          link_left = ln;
        } else {
          cw = rk[0];
          own = reinterpret_cast<const uint4*>(codes)[i];
        }
        if (x + 1 < W) {
          yn = y;
          xn = x + 1;
          cn = rk[kWords];
          on = reinterpret_cast<const uint4*>(codes)[i + 1];
          ln = false;
        }
        if (x + 8 < W && (gl == 0 || gl == 8)) asm volatile("prefetch.global.L1 [%0];" ::"l"(rk + 8 * kWords));
      }
      for (int pass = 0;; ++pass) {
        const int c = static_cast<int>(cw & 255u);
        bool ok = false;
        int at = 0, dj = 0, st = 0;
        if (c != 255 && left > 0) {
          st = step[c];
          at = ci + st;
          if (RING) at += at < 0 ? RW : at >= RW ? -RW : 0;
          dj = count[at];
          const unsigned cc = 0x01010101u * static_cast<unsigned>(c);
          const bool linked = (__vcmpeq4(own.x, cc) | __vcmpeq4(own.y, cc) | __vcmpeq4(own.z, cc) |
                               __vcmpeq4(own.w, cc)) != 0u || (link_left && c == left_code);
          ok = dj < m && !linked;
        }
        const unsigned free16 = __ballot_sync(kAll, ok) >> (lane & 16) & 0xffffu;
        const int n = __popc(free16 & ((1u << gl) - 1u));
        const bool take = ok && n < left;
        if (take) {
          count[at] = static_cast<unsigned char>(dj + 1);
          codes[(i + st) * kMaxM + dj] = static_cast<unsigned char>(NW - 1 - c);  // the way back
          codes[i * kMaxM + dgi + n] = static_cast<unsigned char>(c);
        }
        const unsigned next_linked = __ballot_sync(kAll, take && c == right) >> (lane & 16) & 0xffffu;
        const int last = __shfl_sync(kAll, c, lane | 15);
        ln = ln || next_linked != 0u;
        const int took = min(__popc(free16), left);
        dgi += took;
        left -= took;
        if (last == 255 || pass == kRankPitch / 16 - 1) left = 0;  // the list's end
        if (!__any_sync(kAll, left > 0)) break;
        cw = (pass & 3) != 3 ? cw >> 8 : left > 0 ? rk[(pass + 1) * 4] : kAll;
      }
      if (act && gl == 0) count[ci] = static_cast<unsigned char>(dgi);
    }
    __syncthreads();
  }
  if (RING) {
    const int last = min(H - 1, y0 + rows - 1 + r);
    for (int y = max(first, last - R + 1); y <= last; ++y)
      for (int x = threadIdx.x; x < W; x += blockDim.x) deg[y * W + x] = ring[(y % R) * W + x];
  }
}

// The device tables of the selected links, codes [P][kMaxM] with deg[i] entries:
// sorted neighbour lists nbr [m][P] (-1 padded) and offsets off [m][P].
__global__ void __launch_bounds__(kThreads) k_nl_tables(const unsigned char* __restrict__ codes,
                                                        const unsigned char* __restrict__ deg, int W, int r, int m,
                                                        size_t P, int* __restrict__ nbr, short* __restrict__ off) {
  const size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  if (i >= P) return;
  const int dg = deg[i], side = 2 * r + 1;
  int v[kMaxM];
#pragma unroll
  for (int b = 0; b < kMaxM; ++b) {
    const int c = codes[i * kMaxM + b];
    v[b] = b < dg ? static_cast<int>(i) + (c / side - r) * W + (c % side - r) : 0x7fffffff;
  }
  // odd-even transposition
#pragma unroll
  for (int t = 0; t < kMaxM; ++t)
#pragma unroll
    for (int b = t & 1; b + 1 < kMaxM; b += 2) {
      const int a = min(v[b], v[b + 1]), c = max(v[b], v[b + 1]);
      v[b] = a;
      v[b + 1] = c;
    }
#pragma unroll
  for (int b = 0; b < kMaxM; ++b)
    if (b < m) {
      nbr[b * P + i] = b < dg ? v[b] : -1;
      off[b * P + i] = b < dg ? static_cast<short>(v[b] - static_cast<long long>(i)) : static_cast<short>(0);
    }
}

// rev[b][i]: the position of pixel i in the list of its b-th neighbour.
__global__ void __launch_bounds__(kThreads) k_nl_reverse(const int* __restrict__ nbr, const unsigned char* __restrict__ deg,
                                                         int m, size_t P, unsigned char* __restrict__ rev) {
  const size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  if (i >= P) return;
  const int dg = deg[i];
  for (int b = 0; b < m; ++b) {
    int pos = 0;
    if (b < dg) {
      const size_t j = static_cast<size_t>(nbr[b * P + i]);
      const int dj = deg[j];
      while (pos + 1 < dj && nbr[pos * P + j] != static_cast<int>(i)) ++pos;
    }
    rev[b * P + i] = static_cast<unsigned char>(pos);
  }
}

// The neighbours of pixel i into registers: nb[b] for b < deg(i).
__device__ __forceinline__ int load_nbrs(const int* __restrict__ nbr, const unsigned char* __restrict__ deg, size_t P,
                                         size_t i, int m, int (&nb)[kMaxM]) {
  const int dg = deg[i];
#pragma unroll
  for (int b = 0; b < kMaxM; ++b) nb[b] = (b < dg && b < m) ? nbr[b * P + i] : 0;
  return dg;
}

// One Chebyshev step for (I + D^T D) x = rhs on every label:
// r = rhs - x - 2 (deg x - sum_nbrs x), d <- a d + c r, x_out = x_in + d.
// The iterates, the direction and the right-hand side are pixel-major, four
// labels per float4, so that each neighbour is one 16-byte load per four
// labels; the first step reads u label-major ([K][P], IN_LM) and the last
// also writes it back label-major (OUT_LM).
__device__ __forceinline__ float4 f4_axpy(float a, float4 x, float4 y) {
  return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
}

template <bool IN_LM, bool OUT_LM>
__global__ void __launch_bounds__(kThreads) k_nl_cheb(const float* __restrict__ xin_lm, const float4* __restrict__ xin,
                                                      float* __restrict__ xout_lm, float4* __restrict__ xout,
                                                      float4* __restrict__ d, const float4* __restrict__ rhs,
                                                      const short* __restrict__ off,
                                                      const unsigned char* __restrict__ deg, int K, int Q, int m,
                                                      size_t P, float a, float c) {
  shf::fast::pdl_wait();  // x and d come from the previous step
  shf::fast::pdl_trigger();
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < P;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int dg = deg[i];
    int nb[kMaxM];
#pragma unroll
    for (int b = 0; b < kMaxM; ++b) nb[b] = (b < dg && b < m) ? static_cast<int>(i) + off[b * P + i] : 0;
    auto load = [&](size_t j, int qd) -> float4 {
      if constexpr (IN_LM) {
        const int k0 = 4 * qd;
        return make_float4(xin_lm[k0 * P + j], k0 + 1 < K ? xin_lm[(k0 + 1) * P + j] : 0.f,
                           k0 + 2 < K ? xin_lm[(k0 + 2) * P + j] : 0.f, k0 + 3 < K ? xin_lm[(k0 + 3) * P + j] : 0.f);
      } else {
        return xin[j * Q + qd];
      }
    };
    for (int qd = 0; qd < Q; ++qd) {
      const float4 xi = load(i, qd);
      float4 sn = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int b = 0; b < kMaxM; ++b) {
        if (b < dg) {
          const float4 xn = load(static_cast<size_t>(nb[b]), qd);
          sn = make_float4(sn.x + xn.x, sn.y + xn.y, sn.z + xn.z, sn.w + xn.w);
        }
      }
      const float fd = static_cast<float>(dg);
      const float4 rh = rhs[i * Q + qd];
      const float4 res = make_float4(rh.x - (xi.x + 2.f * (fd * xi.x - sn.x)), rh.y - (xi.y + 2.f * (fd * xi.y - sn.y)),
                                     rh.z - (xi.z + 2.f * (fd * xi.z - sn.z)), rh.w - (xi.w + 2.f * (fd * xi.w - sn.w)));
      const float4 dn = f4_axpy(c, res, make_float4(a * d[i * Q + qd].x, a * d[i * Q + qd].y, a * d[i * Q + qd].z,
                                                     a * d[i * Q + qd].w));
      d[i * Q + qd] = dn;
      const float4 xo = make_float4(xi.x + dn.x, xi.y + dn.y, xi.z + dn.z, xi.w + dn.w);
      if constexpr (OUT_LM) {
        const int k0 = 4 * qd;
        xout_lm[k0 * P + i] = xo.x;
        if (k0 + 1 < K) xout_lm[(k0 + 1) * P + i] = xo.y;
        if (k0 + 2 < K) xout_lm[(k0 + 2) * P + i] = xo.z;
        if (k0 + 3 < K) xout_lm[(k0 + 3) * P + i] = xo.w;
      }
      xout[i * Q + qd] = xo;
    }
  }
}

// The whole Chebyshev solve in one cooperative launch (K <= 4: one float4 per
// pixel), for images whose pixels fit the resident grid.  CTA c owns the
// contiguous pixels [c B, c B + B), B = kChebThreads kChebPPT; each thread
// keeps its pixels' right-hand side, direction d and iterate in registers for
// all the steps, and the CTA keeps its pixels' neighbour offsets (at most MM
// per pixel) in shared memory.  Per step the CTA copies the iterate on the
// window halo of its pixels (R = r W + r pixels on each side: every neighbour
// offset falls inside it) from the previous step's buffer into shared memory
// (asynchronous copies through L2), puts its own pixels there from registers,
// gathers the neighbours there, and writes its pixels to the other buffer; a
// grid barrier separates the steps.  The arithmetic is k_nl_cheb's, in its
// order.
constexpr int kChebPPT = 2;
constexpr int kChebThreads = 1024;
constexpr int kChebBlock = kChebPPT * kChebThreads;         // pixels per CTA
constexpr unsigned long long kBarrierNs = 1000000000ull;  // a barrier gives up after one second

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid barrier number gen (1, 2, ...) on a counter that was zero at launch:
// every CTA adds one and waits until gen * gridDim.x CTAs have arrived.  The
// wait is bounded: after kBarrierNs it sets *err and the barrier reports
// failure (every CTA then leaves the kernel; the host reads *err).
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned gen, int* err) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    // release: the CTA's writes (ordered before this thread by the CTA
    // barrier) become visible with the arrival; acquire on the way out
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    const unsigned target = gen * gridDim.x;
    const unsigned long long t0 = global_ns();
    int ok = 1;
    while (load_acquire(bar) < target) {
      if (global_ns() - t0 > kBarrierNs) {
        ok = 0;
        atomicExch(err, 1);
        break;
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

template <int MM>
__global__ void __launch_bounds__(kChebThreads, 1) k_nl_cheb_all(float* __restrict__ u, float4* xa, float4* xb,
                                                               const float4* __restrict__ rhs,
                                                               const short* __restrict__ off,
                                                               const unsigned char* __restrict__ deg, int K, int m,
                                                               size_t P, int R, int nsteps,
                                                               const float2* __restrict__ ac, unsigned* bar,
                                                               int* err) {
  extern __shared__ __align__(16) float4 sx[];  // the iterate on [lo, hi), then the offsets
  short* so = reinterpret_cast<short*>(sx + kChebBlock + 2 * static_cast<size_t>(R));  // [MM][kChebBlock]
  const size_t base = static_cast<size_t>(blockIdx.x) * kChebBlock;
  const size_t lo = base > static_cast<size_t>(R) ? base - R : 0;
  const size_t hi = base + kChebBlock + R < P ? base + kChebBlock + R : P;
  for (int e = threadIdx.x; e < MM * kChebBlock; e += kChebThreads) {
    const int b = e / kChebBlock, j = e - b * kChebBlock;
    const size_t i = base + j;
    so[e] = (i < P && b < m) ? off[b * P + i] : static_cast<short>(0);
  }
  int dg[kChebPPT];
  float4 r[kChebPPT], dd[kChebPPT], xi[kChebPPT];
#pragma unroll
  for (int p = 0; p < kChebPPT; ++p) {
    const size_t i = base + p * kChebThreads + threadIdx.x;
    const bool live = i < P;
    dg[p] = live ? min(static_cast<int>(deg[i]), m) : 0;
    r[p] = live ? rhs[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    dd[p] = make_float4(0.f, 0.f, 0.f, 0.f);
    xi[p] = live ? make_float4(u[i], K > 1 ? u[P + i] : 0.f, K > 2 ? u[2 * P + i] : 0.f, K > 3 ? u[3 * P + i] : 0.f)
                 : make_float4(0.f, 0.f, 0.f, 0.f);
    if (live) xa[i] = xi[p];
  }
  if (!grid_barrier(bar, 1, err)) return;
  const float4* xin = xa;
  float4* xout = xb;
  for (int k = 0; k < nsteps; ++k) {
    // the halos by asynchronous 16-byte copies (through L2: other CTAs wrote
    // them in the previous step), all in flight at once; the CTA's own
    // pixels from registers
    const size_t own_end = base + kChebBlock < hi ? base + kChebBlock : hi;
    for (size_t j = lo + threadIdx.x; j < hi; j += kChebThreads) {
      if (j >= base && j < own_end) continue;
      const unsigned dst = static_cast<unsigned>(__cvta_generic_to_shared(sx + (j - lo)));
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(xin + j) : "memory");
    }
#pragma unroll
    for (int p = 0; p < kChebPPT; ++p) {
      const size_t i = base + p * kChebThreads + threadIdx.x;
      if (i < P) sx[i - lo] = xi[p];
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const float a = ac[k].x, c = ac[k].y;
#pragma unroll
    for (int p = 0; p < kChebPPT; ++p) {
      const size_t i = base + p * kChebThreads + threadIdx.x;
      if (i >= P) continue;
      const long long il = static_cast<long long>(i - lo);
      const short* sop = so + p * kChebThreads + threadIdx.x;
      float4 sn = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int b = 0; b < MM; ++b) {
        if (b < dg[p]) {
          const float4 xn = sx[il + sop[b * kChebBlock]];
          sn = make_float4(sn.x + xn.x, sn.y + xn.y, sn.z + xn.z, sn.w + xn.w);
        }
      }
      const float fd = static_cast<float>(dg[p]);
      const float4 x = xi[p], rh = r[p], d0 = dd[p];
      const float4 res = make_float4(rh.x - (x.x + 2.f * (fd * x.x - sn.x)), rh.y - (x.y + 2.f * (fd * x.y - sn.y)),
                                     rh.z - (x.z + 2.f * (fd * x.z - sn.z)), rh.w - (x.w + 2.f * (fd * x.w - sn.w)));
      const float4 dn = f4_axpy(c, res, make_float4(a * d0.x, a * d0.y, a * d0.z, a * d0.w));
      dd[p] = dn;
      xi[p] = make_float4(x.x + dn.x, x.y + dn.y, x.z + dn.z, x.w + dn.w);
      if (k + 1 < nsteps) xout[i] = xi[p];
    }
    if (k + 1 < nsteps) {
      if (!grid_barrier(bar, static_cast<unsigned>(k) + 2u, err)) return;  // also orders the shared reads
      const float4* t = xout;
      xout = const_cast<float4*>(xin);
      xin = t;
    }
  }
#pragma unroll
  for (int p = 0; p < kChebPPT; ++p) {
    const size_t i = base + p * kChebThreads + threadIdx.x;
    if (i >= P) continue;
    xout[i] = xi[p];  // nobody reads that buffer in the last step
    u[i] = xi[p].x;
    if (K > 1) u[P + i] = xi[p].y;
    if (K > 2) u[2 * P + i] = xi[p].z;
    if (K > 3) u[3 * P + i] = xi[p].w;
  }
}

// The barrier with a target no CTA reaches (each arrives once, generation 2
// needs two arrivals each): the bounded wait must give up (self-test).
__global__ void k_barrier_unreachable(unsigned* bar, int* err) { grid_barrier(bar, 2, err); }

// Shared memory of the persistent solve: the iterate on the CTA's pixels and
// two halos, and MM neighbour offsets per pixel.
size_t cheb_all_smem(int R, int MM) {
  return sizeof(float4) * (static_cast<size_t>(kChebBlock) + 2 * static_cast<size_t>(R)) +
         sizeof(short) * static_cast<size_t>(MM) * kChebBlock;
}

// The v-, w- and b-updates after the u-step: g_b = b_v,b + u(nbr_b) - u(i)
// (b < deg; b_v,b for the zero rows), group clip over the m K values,
// d = g - 2 b_v; w-step and q = (w - b_w) - gamma s.  xu: u pixel-major.
// With four labels per float4 a neighbour is one 16-byte load (the labels one
// by one took four 4-byte loads each, of sectors that held nothing else), and
// for K <= 4 (ONE) all g of a pixel stay in registers between the norm and the
// update; otherwise they are formed twice.  MM: at most m neighbours (10 for
// the paper's five picked per pixel).  Bound by memory: per pixel 3 m Q 16 B of
// b_v and d, 150 MB at 512 x 512, K = 4, m = 10: 112 -> 44 us.
template <int KM, int MM, bool ONE>
__global__ void __launch_bounds__(kThreads) k_nl_prox(const float4* __restrict__ xu, float4* __restrict__ bv,
                                                      float4* __restrict__ d, float* __restrict__ w,
                                                      float* __restrict__ bw, const float* __restrict__ s,
                                                      float4* __restrict__ q, const short* __restrict__ off,
                                                      const unsigned char* __restrict__ deg, int K, int Q, int m,
                                                      size_t P, float t, float gamma) {
  shf::fast::pdl_wait();  // u comes from the last Chebyshev step
  shf::fast::pdl_trigger();
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < P;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int dg = deg[i];
    int nb[MM];
#pragma unroll
    for (int b = 0; b < MM; ++b) nb[b] = b < dg ? static_cast<int>(i) + off[b * P + i] : static_cast<int>(i);
    auto diff = [&](int b, int qd, float4 ui) {  // g_b; the pixel itself stands in for a missing neighbour
      const float4 x = xu[static_cast<size_t>(nb[b]) * Q + qd];
      const float4 o = bv[(static_cast<size_t>(qd) * m + b) * P + i];
      return make_float4(o.x + (x.x - ui.x), o.y + (x.y - ui.y), o.z + (x.z - ui.z), o.w + (x.w - ui.w));
    };
    float4 g[ONE ? MM : 1];
    float n2 = 0.f;
    for (int qd = 0; qd < (ONE ? 1 : Q); ++qd) {
      const float4 ui = xu[i * Q + qd];
#pragma unroll
      for (int b = 0; b < MM; ++b) {
        if (b < m) {
          const float4 v = diff(b, qd, ui);
          if (ONE) g[ONE ? b : 0] = v;
          n2 = fmaf(v.x, v.x, n2);
          n2 = fmaf(v.y, v.y, n2);
          n2 = fmaf(v.z, v.z, n2);
          n2 = fmaf(v.w, v.w, n2);
        }
      }
    }
    const float nrm = sqrtf(n2);
    const float fac = nrm > t ? t / nrm : 1.f;
    for (int qd = 0; qd < (ONE ? 1 : Q); ++qd) {
      const float4 ui = xu[i * Q + qd];
#pragma unroll
      for (int b = 0; b < MM; ++b) {
        if (b < m) {
          const float4 v = ONE ? g[ONE ? b : 0] : diff(b, qd, ui);
          const float4 bn = make_float4(fac * v.x, fac * v.y, fac * v.z, fac * v.w);
          bv[(static_cast<size_t>(qd) * m + b) * P + i] = bn;
          d[(static_cast<size_t>(qd) * m + b) * P + i] =
              make_float4(v.x - 2.f * bn.x, v.y - 2.f * bn.y, v.z - 2.f * bn.z, v.w - 2.f * bn.w);
        }
      }
    }
    float gw[KM], wk[KM];
#pragma unroll
    for (int k = 0; k < KM; k += 4) {
      const float4 ui = k < K ? xu[i * Q + k / 4] : make_float4(0.f, 0.f, 0.f, 0.f);
      const float uk[4] = {ui.x, ui.y, ui.z, ui.w};
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        gw[k + c] = k + c < K ? bw[(k + c) * P + i] + uk[c] : 0.f;
        wk[k + c] = gw[k + c];
      }
    }
    shf::simplex_project_sorted<KM>(wk, K);
#pragma unroll
    for (int k = 0; k < KM; k += 4) {
      float qv[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (k + c < K) {
          const float bn = gw[k + c] - wk[k + c];
          w[(k + c) * P + i] = wk[k + c];
          bw[(k + c) * P + i] = bn;
          qv[c] = (wk[k + c] - bn) - gamma * s[(k + c) * P + i];
        }
      if (k < K) q[i * Q + k / 4] = make_float4(qv[0], qv[1], qv[2], qv[3]);
    }
  }
}

// rhs = q + D^T d: (D^T d)(j) = sum_{b < deg(j)} [d_rev(j,b)(nbr_b(j)) - d_b(j)],
// pixel-major as the Chebyshev steps read it (512 x 512, K = 4: 47 -> 27 us with
// one 16-byte load per neighbour).
template <int MM>
__global__ void __launch_bounds__(kThreads) k_nl_rhs(const float4* __restrict__ q, const float4* __restrict__ d,
                                                     float4* __restrict__ rhs, const short* __restrict__ off,
                                                     const unsigned char* __restrict__ rev,
                                                     const unsigned char* __restrict__ deg, int Q, int m, size_t P) {
  shf::fast::pdl_wait();  // q and d come from the prox kernel
  shf::fast::pdl_trigger();
  for (size_t j = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; j < P;
       j += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int dg = deg[j];
    size_t at[MM];  // where the neighbour keeps its difference to j
#pragma unroll
    for (int b = 0; b < MM; ++b)
      at[b] = b < dg ? static_cast<size_t>(rev[b * P + j]) * P + (static_cast<long long>(j) + off[b * P + j]) : 0;
    for (int qd = 0; qd < Q; ++qd) {
      const float4* dq = d + static_cast<size_t>(qd) * m * P;
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int b = 0; b < MM; ++b)
        if (b < dg) {
          const float4 x = dq[at[b]], y = dq[b * P + j];
          acc = make_float4(acc.x + (x.x - y.x), acc.y + (x.y - y.y), acc.z + (x.z - y.z), acc.w + (x.w - y.w));
        }
      const float4 qv = q[j * Q + qd];
      rhs[j * Q + qd] = make_float4(qv.x + acc.x, qv.y + acc.y, qv.z + acc.z, qv.w + acc.w);
    }
  }
}

// q from label-major planes, pixel-major.
__global__ void k_nl_q(const float* __restrict__ w, const float* __restrict__ bw, const float* __restrict__ s,
                       float* __restrict__ q, float gamma, int K, int Q, size_t P) {
  const size_t n = P * 4 * Q;
  for (size_t e = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; e < n;
       e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t i = e / (4 * Q), k = e - i * 4 * Q;
    q[e] = k < static_cast<size_t>(K) ? (w[k * P + i] - bw[k * P + i]) - gamma * s[k * P + i] : 0.f;
  }
}

// The neighbour pairs of the state ([Q][m][P] float4) as label-major planes
// [K][m][P]: out = a + sb b (b optional), and back: out = a + sb b with a
// label-major, labels past K zero.
__global__ void k_nl_unpack(const float4* __restrict__ a, const float4* __restrict__ b, float* __restrict__ out, float sb,
                            int K, int Q, size_t mP) {
  for (size_t e = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; e < mP * Q;
       e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t qd = e / mP, i = e - qd * mP;
    const float4 x = a[e], y = b ? b[e] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float v[4] = {x.x + sb * y.x, x.y + sb * y.y, x.z + sb * y.z, x.w + sb * y.w};
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (4 * qd + c < static_cast<size_t>(K)) out[(4 * qd + c) * mP + i] = v[c];
  }
}
__global__ void k_nl_pack(const float* __restrict__ a, const float4* __restrict__ b, float4* __restrict__ out, float sb,
                          int K, int Q, size_t mP) {
  for (size_t e = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; e < mP * Q;
       e += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const size_t qd = e / mP, i = e - qd * mP;
    const float4 y = b ? b[e] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float o[4] = {y.x, y.y, y.z, y.w};
    float v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const size_t k = 4 * qd + c;
      v[c] = k < static_cast<size_t>(K) ? a[k * mP + i] + sb * o[c] : 0.f;
    }
    out[e] = make_float4(v[0], v[1], v[2], v[3]);
  }
}

// FP64 energy partials: <w, s> and sum_i (sum_k sum_b ((D w_k)_b(i))^2)^(1/2).
__global__ void __launch_bounds__(kThreads) k_nl_energy(const float* __restrict__ w, const float* __restrict__ s,
                                                        const int* __restrict__ nbr,
                                                        const unsigned char* __restrict__ deg, int K, int m, size_t P,
                                                        double* __restrict__ partial) {
  double ds = 0.0, dt = 0.0;
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < P;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    int nb[kMaxM];
    const int dg = load_nbrs(nbr, deg, P, i, m, nb);
    double n2 = 0.0;
    for (int k = 0; k < K; ++k) {
      const float* wp = w + k * P;
      ds += static_cast<double>(wp[i]) * s[k * P + i];
#pragma unroll
      for (int b = 0; b < kMaxM; ++b) {
        if (b < dg) {
          const double e = static_cast<double>(wp[nb[b]]) - wp[i];
          n2 += e * e;
        }
      }
    }
    dt += sqrt(n2);
  }
  __shared__ double sh[2][kThreads];
  sh[0][threadIdx.x] = ds;
  sh[1][threadIdx.x] = dt;
  __syncthreads();
  for (int o = kThreads / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + o];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    partial[2 * blockIdx.x] = sh[0][0];
    partial[2 * blockIdx.x + 1] = sh[1][0];
  }
}

__global__ void k_nl_energy_final(const double* __restrict__ partial, int nblocks, double* __restrict__ out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double a = 0.0, b = 0.0;
  for (int i = 0; i < nblocks; ++i) {
    a += partial[2 * i];
    b += partial[2 * i + 1];
  }
  out[0] = a;
  out[1] = b;
}

int nl_fail(int code, const std::string& msg) { return shf::set_error(code, msg); }

#define NL_CK(call)                                                                                         \
  do {                                                                                                      \
    cudaError_t e_ = (call);                                                                                \
    if (e_ != cudaSuccess) return nl_fail(SHF_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

template <typename T>
int nl_alloc(T** p, size_t count, const char* what) {
  *p = nullptr;
  if (count == 0) return SHF_OK;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), count * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return nl_fail(e == cudaErrorMemoryAllocation ? SHF_ERR_OOM : SHF_ERR_CUDA,
                   std::string("cudaMalloc(") + what + "): " + cudaGetErrorString(e));
  }
  return SHF_OK;
}

// Pinned host memory: the graph's copies run at the link's rate and touch no new
// pages on a reset.
template <typename T>
int nl_alloc_host(T** p, size_t count, const char* what) {
  *p = nullptr;
  cudaError_t e = cudaMallocHost(reinterpret_cast<void**>(p), count * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return nl_fail(e == cudaErrorMemoryAllocation ? SHF_ERR_OOM : SHF_ERR_CUDA,
                   std::string("cudaMallocHost(") + what + "): " + cudaGetErrorString(e));
  }
  return SHF_OK;
}

int grid_for(size_t n) {
  const size_t b = (n + kThreads - 1) / kThreads;
  return static_cast<int>(b < 8192 ? (b ? b : 1) : 8192);
}

void free_nl(nl_state* st) {
  if (!st) return;
  if (st->stream) cudaStreamSynchronize(st->stream);
  if (st->exec) cudaGraphExecDestroy(st->exec);
  void* bufs[] = {st->f, st->s, st->u, st->xa, st->xb, st->cd, st->bv, st->d, st->w, st->bw, st->q, st->rhs,
                  st->gap, st->nbr, st->off, st->rev, st->deg, st->gw, st->rank, st->codes, st->labels, st->flag,
                  st->red,
                  st->cbar, st->cerr, st->cheb_ac};
  for (void* b : bufs) cudaFree(b);
  cudaFreeHost(st->codes_host);
  cudaFreeHost(st->deg_host);
  if (st->own_stream && st->stream) cudaStreamDestroy(st->stream);
  delete st;
}

// Patch weights G_a on the (2h+1)^2 patch, normalised to sum 1.
std::vector<double> patch_weights(int h, double a) {
  const int n = 2 * h + 1;
  std::vector<double> G(static_cast<size_t>(n) * n);
  double sum = 0.0;
  for (int t1 = -h; t1 <= h; ++t1)
    for (int t2 = -h; t2 <= h; ++t2) {
      const double g = std::exp(-static_cast<double>(t1 * t1 + t2 * t2) / (2.0 * a * a));
      G[(t1 + h) * n + (t2 + h)] = g;
      sum += g;
    }
  for (double& g : G) g /= sum;
  return G;
}

// The graph of st->f: ranks and selection, the device tables (neighbours [m][P],
// reverse positions, counts), the links on the host, and the Chebyshev
// coefficients.  Synchronises.
int build_graph(nl_state* st) {
  const int H = st->H, W = st->W, mt = st->prm.neighbours, m = st->m;
  const int h = st->prm.patch / 2, r = st->prm.window / 2, side = 2 * r + 1;
  const size_t P = st->P();
  const auto G = patch_weights(h, st->prm.a);
  // twice the FP32 distances' relative error bound; negative when a weight is
  // too small for it
  double gmin = G[0];
  for (double g : G) gmin = std::min(gmin, g);
  const float bound = gmin < 1e-30 ? -1.f : static_cast<float>(2.02 * (static_cast<double>(G.size()) * st->C + 4) / 16777216.0);
  NL_CK(cudaMemcpyAsync(st->gw, G.data(), sizeof(double) * G.size(), cudaMemcpyHostToDevice, st->stream));
  auto* codes = reinterpret_cast<unsigned char*>(st->codes);
  const auto* rank = reinterpret_cast<const unsigned*>(st->rank);
  NL_CK(cudaMemsetAsync(codes, 255, P * kMaxM, st->stream));
  NL_CK(cudaMemsetAsync(st->deg, 0, P, st->stream));
  for (int y = 0; y < H; y += st->rank_rows) {
    const int rows = std::min(st->rank_rows, H - y);
    const dim3 grid((W + kRankTX - 1) / kRankTX, (rows + kRankTY - 1) / kRankTY);
    if (st->C == 1)
      k_nl_rank<1><<<grid, 32 * kRankWarps, 0, st->stream>>>(st->f, H, W, st->gw, h, r, bound, y, y + rows, st->rank);
    else
      k_nl_rank<3><<<grid, 32 * kRankWarps, 0, st->stream>>>(st->f, H, W, st->gw, h, r, bound, y, y + rows, st->rank);
    NL_CK(cudaGetLastError());
    // a half warp for every row of a step
    const int threads = std::min(1024, (std::min(rows, (W + side - 1) / side) + 1) / 2 * 32);
    const int R = 2 * r + (W - 1) / side + 1;
    if (static_cast<size_t>(R) * W <= kRingBytes) {
      NL_CK(cudaFuncSetAttribute(k_nl_select<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kRingBytes)));
      k_nl_select<true><<<1, threads, static_cast<size_t>(R) * W, st->stream>>>(rank, H, W, r, m, mt, y, rows, R, codes, st->deg);
    } else {
      k_nl_select<false><<<1, threads, 0, st->stream>>>(rank, H, W, r, m, mt, y, rows, R, codes, st->deg);
    }
    NL_CK(cudaGetLastError());
  }
  const unsigned tgrid = static_cast<unsigned>((P + kThreads - 1) / kThreads);
  k_nl_tables<<<tgrid, kThreads, 0, st->stream>>>(codes, st->deg, W, r, m, P, st->nbr, st->off);
  NL_CK(cudaGetLastError());
  k_nl_reverse<<<tgrid, kThreads, 0, st->stream>>>(st->nbr, st->deg, m, P, st->rev);
  NL_CK(cudaGetLastError());
  NL_CK(cudaMemcpyAsync(st->codes_host, codes, P * kMaxM, cudaMemcpyDeviceToHost, st->stream));
  NL_CK(cudaMemcpyAsync(st->deg_host, st->deg, P, cudaMemcpyDeviceToHost, st->stream));
  NL_CK(cudaStreamSynchronize(st->stream));
  const unsigned char* const dg = st->deg_host;
  st->deg_max = 0;
  for (size_t i = 0; i < P; ++i) st->deg_max = std::max(st->deg_max, static_cast<int>(dg[i]));
  // Chebyshev iteration on [1, 1 + 4 deg_max]: theta = centre, delta = half width
  const double lo = 1.0, hi = 1.0 + 4.0 * st->deg_max;
  const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo);
  int n = st->prm.solve_steps;
  if (n <= 0) {
    const double kappa = hi / lo;
    const double qrate = (std::sqrt(kappa) - 1.0) / (std::sqrt(kappa) + 1.0);
    n = qrate > 0.0 ? static_cast<int>(std::ceil(std::log(2.0 / 1e-7) / -std::log(qrate))) : 1;
  }
  n = std::max(n + (n & 1), 2);  // even and >= 2: the first step reads u, the last writes it
  st->cheb_a.assign(n, 0.f);
  st->cheb_c.assign(n, 0.f);
  st->cheb_c[0] = static_cast<float>(1.0 / theta);
  if (delta > 0.0) {
    const double sigma = theta / delta;
    double rho = 1.0 / sigma;
    for (int k = 1; k < n; ++k) {
      const double rn = 1.0 / (2.0 * sigma - rho);
      st->cheb_a[k] = static_cast<float>(rn * rho);
      st->cheb_c[k] = static_cast<float>(2.0 * rn / delta);
      rho = rn;
    }
  }
  // the persistent solve: the steps' (a, c) on the device, and its grid when
  // the pixels fit the resident CTAs at kChebPPT pixels per thread
  cudaFree(st->cheb_ac);
  st->cheb_ac = nullptr;
  st->cheb_grid = 0;
  // (the neighbours of a pixel lie in its window: |offset| <= r W + r)
  int coop = 0, sms = 0, per_sm = 0, optin = 0;
  st->cheb_halo = r * W + r;
  const int MM = m <= 10 ? 10 : kMaxM;
  const size_t smem = cheb_all_smem(st->cheb_halo, MM);
  const void* kern = MM == 10 ? reinterpret_cast<const void*>(k_nl_cheb_all<10>)
                              : reinterpret_cast<const void*>(k_nl_cheb_all<kMaxM>);
  if (st->Q == 1 && cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, st->device) == cudaSuccess && coop &&
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, st->device) == cudaSuccess &&
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, st->device) == cudaSuccess &&
      smem <= static_cast<size_t>(optin) &&
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) == cudaSuccess &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kChebThreads, smem) == cudaSuccess) {
    const size_t need = (P + kChebBlock - 1) / kChebBlock;
    if (need >= 1 && need <= static_cast<size_t>(per_sm) * sms) {
      std::vector<float2> ac(n);
      for (int k = 0; k < n; ++k) ac[k] = make_float2(st->cheb_a[k], st->cheb_c[k]);
      int rc = nl_alloc(&st->cheb_ac, static_cast<size_t>(n), "chebyshev coefficients");
      if (rc) return rc;
      NL_CK(cudaMemcpy(st->cheb_ac, ac.data(), sizeof(float2) * n, cudaMemcpyHostToDevice));
      st->cheb_grid = static_cast<int>(need);
    }
  }
  cudaGetLastError();
  return SHF_OK;
}

enum NlKind { kNlSolve = 0, kNlProx = 1, kNlRhs = 2, kNlKinds = 3 };
const char* const kNlNames[kNlKinds] = {"nl_solve", "nl_prox", "nl_rhs"};

// u pixel-major after the solve: the buffer its last step wrote.
const float4* solved(const nl_state* st) { return st->cheb_grid > 0 ? st->xa : st->xb; }

template <int KM, bool ONE>
cudaError_t launch_prox_t(nl_state* st) {
  const auto kern = st->m <= 10 ? k_nl_prox<KM, 10, ONE> : k_nl_prox<KM, kMaxM, ONE>;
  return shf::fast::launch_pdl(kern, dim3(grid_for(st->P())), dim3(kThreads), 0, st->stream, solved(st), st->bv, st->d,
                               st->w, st->bw, st->s, st->q, st->off, st->deg, st->K, st->Q, st->m, st->P(),
                               st->gamma * st->lambda, st->gamma);
}

cudaError_t launch_prox(nl_state* st) {
  if (st->K <= 4) return launch_prox_t<4, true>(st);
  return st->K <= 8 ? launch_prox_t<8, false>(st) : launch_prox_t<16, false>(st);
}

cudaError_t launch_rhs(nl_state* st) {
  return shf::fast::launch_pdl(st->m <= 10 ? k_nl_rhs<10> : k_nl_rhs<kMaxM>, dim3(grid_for(st->P())), dim3(kThreads), 0,
                               st->stream, st->q, st->d, st->rhs, st->off, st->rev, st->deg, st->Q, st->m, st->P());
}

// One iteration; ev (nullable, kNlKinds + 1 events) recorded before each
// part and after the last.
cudaError_t enqueue_nl_iteration(nl_state* st, cudaEvent_t* ev) {
  cudaStream_t ss = st->stream;
  auto mark = [&](int i) { return ev ? cudaEventRecord(ev[i], ss) : cudaSuccess; };
  cudaError_t e = mark(kNlSolve);
  const size_t P = st->P();
  const int n = static_cast<int>(st->cheb_a.size());  // even, >= 2
  float4* x0 = st->xa;
  float4* x1 = st->xb;
  if (st->cheb_grid > 0 && e == cudaSuccess) {  // one cooperative launch for all the steps
    e = cudaMemsetAsync(st->cbar, 0, sizeof(unsigned), ss);
    if (e == cudaSuccess) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(st->cheb_grid);
      cfg.blockDim = dim3(kChebThreads);
      const int MM = st->m <= 10 ? 10 : kMaxM;
      cfg.dynamicSmemBytes = cheb_all_smem(st->cheb_halo, MM);
      cfg.stream = ss;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeCooperative;
      attr[0].val.cooperative = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      e = cudaLaunchKernelEx(&cfg, MM == 10 ? k_nl_cheb_all<10> : k_nl_cheb_all<kMaxM>, st->u, x0, x1, static_cast<const float4*>(st->rhs),
                             static_cast<const short*>(st->off), static_cast<const unsigned char*>(st->deg), st->K,
                             st->m, P, st->cheb_halo, n, static_cast<const float2*>(st->cheb_ac), st->cbar,
                             st->cerr);
    }
  }
  for (int k = 0; k < n && e == cudaSuccess && st->cheb_grid == 0; ++k) {
    const float a = st->cheb_a[k], c = st->cheb_c[k];
    const dim3 grid(grid_for(P)), block(kThreads);
    const float* none = nullptr;
    float* none_out = nullptr;
    const float4* none4 = nullptr;
    if (k == 0)  // from u (label-major)
      e = shf::fast::launch_pdl(k_nl_cheb<true, false>, grid, block, 0, ss, st->u, none4, none_out, x0, st->cd,
                                st->rhs, st->off, st->deg, st->K, st->Q, st->m, P, a, c);
    else if (k == n - 1)  // back into u
      e = shf::fast::launch_pdl(k_nl_cheb<false, true>, grid, block, 0, ss, none, x0, st->u, x1, st->cd,
                                st->rhs, st->off, st->deg, st->K, st->Q, st->m, P, a, c);
    else {
      e = shf::fast::launch_pdl(k_nl_cheb<false, false>, grid, block, 0, ss, none, x0, none_out, x1, st->cd,
                                st->rhs, st->off, st->deg, st->K, st->Q, st->m, P, a, c);
      std::swap(x0, x1);
    }
  }
  if (e == cudaSuccess) e = mark(kNlProx);
  if (e == cudaSuccess) e = launch_prox(st);
  if (e == cudaSuccess) e = mark(kNlRhs);
  if (e == cudaSuccess) e = launch_rhs(st);
  if (e == cudaSuccess) e = mark(kNlKinds);
  return e;
}

cudaError_t rebuild_rhs(nl_state* st) {
  k_nl_q<<<grid_for(st->P() * 4 * st->Q), kThreads, 0, st->stream>>>(st->w, st->bw, st->s, reinterpret_cast<float*>(st->q),
                                                                     st->gamma, st->K, st->Q, st->P());
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? launch_rhs(st) : e;
}

// Graph, data term and the zero state.  Synchronises.
int nl_restart(nl_state* st) {
  const size_t P = st->P(), K = st->K, m = st->m;
  NL_CK(cudaMemsetAsync(st->flag, 0, sizeof(int), st->stream));
  NL_CK(shf::launch_count_nonfinite(st->f, static_cast<long>(P * st->C), st->flag, st->stream));
  int bad = 0;
  NL_CK(cudaMemcpyAsync(&bad, st->flag, sizeof(int), cudaMemcpyDeviceToHost, st->stream));
  NL_CK(cudaStreamSynchronize(st->stream));
  if (bad) return nl_fail(SHF_ERR_NONFINITE, "nl: the image contains NaN or Inf");
  int rc = build_graph(st);
  if (rc) return rc;
  if (st->exec) {  // the step count may have changed with the graph
    cudaGraphExecDestroy(st->exec);
    st->exec = nullptr;
    st->graph_tried = false;
  }
  NL_CK(shf::launch_data_term(st->f, st->C, st->codebook.data(), st->K, st->s, static_cast<int>(P), st->stream));
  NL_CK(cudaMemsetAsync(st->u, 0, sizeof(float) * P * K, st->stream));
  NL_CK(cudaMemsetAsync(st->w, 0, sizeof(float) * P * K, st->stream));
  NL_CK(cudaMemsetAsync(st->bw, 0, sizeof(float) * P * K, st->stream));
  NL_CK(cudaMemsetAsync(st->bv, 0, sizeof(float4) * m * P * st->Q, st->stream));
  NL_CK(cudaMemsetAsync(st->d, 0, sizeof(float4) * m * P * st->Q, st->stream));
  NL_CK(cudaMemsetAsync(st->cd, 0, sizeof(float4) * P * st->Q, st->stream));
  NL_CK(rebuild_rhs(st));
  NL_CK(cudaStreamSynchronize(st->stream));
  st->iter = 0;
  return SHF_OK;
}

int nl_copy(nl_state* st, void* dst, const void* src, size_t bytes, cudaMemcpyKind kind, bool sync) {
  NL_CK(cudaMemcpyAsync(dst, src, bytes, kind, st->stream));
  if (sync) NL_CK(cudaStreamSynchronize(st->stream));
  return SHF_OK;
}

}  // namespace

extern "C" {

int nl_admm_init(int H, int W, const float* f, int C, const float* codebook, int K, const nl_params* p, void* stream,
                 nl_state** out) {
  if (!out) return nl_fail(SHF_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (!f || !codebook || !p) return nl_fail(SHF_ERR_ARG, "nl_admm_init: NULL argument");
  if (K < 2 || K > shf::kMaxK) return nl_fail(SHF_ERR_ARG, "K must be in [2, 16]");
  if (C != 1 && C != 3) return nl_fail(SHF_ERR_ARG, "C must be 1 or 3");
  if (!(p->gamma > 0.f) || !std::isfinite(p->gamma)) return nl_fail(SHF_ERR_ARG, "gamma must be positive and finite");
  if (!(p->lambda >= 0.f) || !std::isfinite(p->lambda))
    return nl_fail(SHF_ERR_ARG, "lambda must be finite and non-negative");
  if (p->patch < 1 || p->patch > kMaxPatch) return nl_fail(SHF_ERR_ARG, "patch must be in [1, 9]");
  if (p->window < 3 || p->window > kMaxWin || !(p->window & 1)) return nl_fail(SHF_ERR_ARG, "window must be odd, 3..15");
  if (!(p->a > 0.f) || !std::isfinite(p->a)) return nl_fail(SHF_ERR_ARG, "a must be positive");
  if (p->neighbours < 1 || 2 * p->neighbours > kMaxM) return nl_fail(SHF_ERR_ARG, "neighbours must be in [1, 8]");
  if (p->solve_steps < 0 || p->solve_steps > 1000) return nl_fail(SHF_ERR_ARG, "solve_steps must be in [0, 1000]");
  if (H < 8 || W < 8 || H > shf::kMaxSide || W > shf::kMaxSide) return nl_fail(SHF_ERR_SIZE, "H and W must be in [8, 2048]");
  if (reinterpret_cast<uintptr_t>(f) & 7u) return nl_fail(SHF_ERR_ARG, "f must be 8-byte aligned");
  for (int i = 0; i < K * C; ++i)
    if (!std::isfinite(codebook[i])) return nl_fail(SHF_ERR_NONFINITE, "codebook contains NaN or Inf");
  auto* st = new nl_state();
  st->H = H;
  st->W = W;
  st->K = K;
  st->C = C;
  st->prm = *p;
  st->m = 2 * p->neighbours;
  st->Q = (K + 3) / 4;
  st->gamma = p->gamma;
  st->lambda = p->lambda;
  st->codebook.assign(codebook, codebook + K * C);
  cudaError_t ed = cudaGetDevice(&st->device);
  if (ed != cudaSuccess) {
    delete st;
    return nl_fail(SHF_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(ed));
  }
  if (stream) {
    st->stream = static_cast<cudaStream_t>(stream);
  } else {
    cudaError_t e = cudaStreamCreateWithFlags(&st->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
      delete st;
      return nl_fail(SHF_ERR_CUDA, std::string("cudaStreamCreate: ") + cudaGetErrorString(e));
    }
    st->own_stream = true;
  }
  const size_t P = static_cast<size_t>(H) * W, m = st->m;
  const size_t rank_row = static_cast<size_t>(W) * kRankPitch;
  st->rank_rows = static_cast<int>(std::min<size_t>(H, std::max<size_t>(kRankBytes / rank_row, kRankTY)));
  int rc;
  if ((rc = nl_alloc(&st->f, P * C, "f")) || (rc = nl_alloc(&st->s, P * K, "s")) ||
      (rc = nl_alloc(&st->u, P * K, "u")) || (rc = nl_alloc(&st->xa, P * st->Q, "chebyshev x")) ||
      (rc = nl_alloc(&st->xb, P * st->Q, "chebyshev x")) || (rc = nl_alloc(&st->cd, P * st->Q, "chebyshev d")) ||
      (rc = nl_alloc(&st->bv, m * P * st->Q, "b_v")) ||
      (rc = nl_alloc(&st->d, m * P * st->Q, "d")) || (rc = nl_alloc(&st->w, P * K, "w")) ||
      (rc = nl_alloc(&st->bw, P * K, "b_w")) || (rc = nl_alloc(&st->q, P * st->Q, "q")) ||
      (rc = nl_alloc(&st->rhs, P * st->Q, "rhs")) || (rc = nl_alloc(&st->gap, P, "gap")) ||
      (rc = nl_alloc(&st->nbr, P * m, "neighbours")) || (rc = nl_alloc(&st->off, P * m, "offsets")) ||
      (rc = nl_alloc(&st->rev, P * m, "reverse")) || (rc = nl_alloc(&st->gw, kMaxPatch * kMaxPatch, "weights")) ||
      (rc = nl_alloc(&st->codes, P, "links")) ||
      (rc = nl_alloc_host(&st->codes_host, P * kMaxM, "links")) || (rc = nl_alloc_host(&st->deg_host, P, "counts")) ||
      (rc = nl_alloc(&st->deg, P, "counts")) || (rc = nl_alloc(&st->labels, P, "labels")) ||
      (rc = nl_alloc(&st->flag, 1, "flag")) || (rc = nl_alloc(&st->red, 2 * kRedBlocks + 2, "red")) ||
      (rc = nl_alloc(&st->cbar, 1, "barrier")) || (rc = nl_alloc(&st->cerr, 1, "barrier flag"))) {
    free_nl(st);
    return rc;
  }
  // as many rows' ranks at a time as there is memory for
  while ((rc = nl_alloc(&st->rank, rank_row * st->rank_rows, "ranks")) == SHF_ERR_OOM && st->rank_rows > kRankTY)
    st->rank_rows = std::max(kRankTY, st->rank_rows / 2);
  if (rc) {
    free_nl(st);
    return rc;
  }
  if (cudaMemset(st->cerr, 0, sizeof(int)) != cudaSuccess) {
    free_nl(st);
    return nl_fail(SHF_ERR_CUDA, "nl_admm_init: cudaMemset");
  }
  cudaError_t e = cudaMemcpyAsync(st->f, f, sizeof(float) * P * C, cudaMemcpyDeviceToDevice, st->stream);
  if (e != cudaSuccess) {
    free_nl(st);
    return nl_fail(SHF_ERR_CUDA, std::string("nl_admm_init: ") + cudaGetErrorString(e));
  }
  rc = nl_restart(st);
  if (rc) {
    free_nl(st);
    return rc;
  }
  *out = st;
  return SHF_OK;
}

int nl_admm_reset(nl_state* st, const float* f, int f_on_host) {
  if (!st || !f) return nl_fail(SHF_ERR_ARG, "nl_admm_reset: NULL argument");
  if (!f_on_host && (reinterpret_cast<uintptr_t>(f) & 7u)) return nl_fail(SHF_ERR_ARG, "f must be 8-byte aligned");
  NL_CK(cudaMemcpyAsync(st->f, f, sizeof(float) * st->P() * st->C,
                        f_on_host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, st->stream));
  return nl_restart(st);
}

int nl_admm_graph(const nl_state* st, int* nbr, int* deg, int* solve_steps) {
  if (!st) return nl_fail(SHF_ERR_ARG, "nl_admm_graph: NULL state");
  if (nbr) {  // the selection's links, sorted, -1 padded
    const size_t P = st->P(), m = st->m;
    const int side = 2 * (st->prm.window / 2) + 1, r = side / 2;
    for (size_t i = 0; i < P; ++i) {
      int* o = nbr + i * m;
      for (int b = 0; b < st->deg_host[i]; ++b) {
        const int c = st->codes_host[i * kMaxM + b];
        o[b] = static_cast<int>(i) + (c / side - r) * st->W + (c % side - r);
      }
      std::sort(o, o + st->deg_host[i]);
      std::fill(o + st->deg_host[i], o + m, -1);
    }
  }
  if (deg) std::copy(st->deg_host, st->deg_host + st->P(), deg);
  if (solve_steps) *solve_steps = static_cast<int>(st->cheb_a.size());
  return SHF_OK;
}

int nl_admm_step(nl_state* st, int n) {
  if (!st || n < 0) return nl_fail(SHF_ERR_ARG, "nl_admm_step: bad argument");
  if (n == 0) return SHF_OK;
  if (!st->graph_tried) {
    st->graph_tried = true;
    cudaGraph_t graph = nullptr;
    if (st->stream && cudaStreamBeginCapture(st->stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
      cudaError_t e = enqueue_nl_iteration(st, nullptr);
      cudaError_t e2 = cudaStreamEndCapture(st->stream, &graph);
      if (e == cudaSuccess && e2 == cudaSuccess && graph) {
        if (cudaGraphInstantiate(&st->exec, graph, 0) != cudaSuccess) st->exec = nullptr;
      }
      if (graph) cudaGraphDestroy(graph);
    }
    cudaGetLastError();  // also of a stream that can't be captured
  }
  for (int i = 0; i < n; ++i) {
    if (st->exec)
      NL_CK(cudaGraphLaunch(st->exec, st->stream));
    else
      NL_CK(enqueue_nl_iteration(st, nullptr));
  }
  st->iter += n;
  return SHF_OK;
}

int nl_admm_kernel_times(nl_state* st, int n, float* ms, int* nk) {
  if (!st || !ms || n < 1) return nl_fail(SHF_ERR_ARG, "nl_admm_kernel_times: bad argument");
  cudaEvent_t ev[kNlKinds + 1];
  for (int i = 0; i <= kNlKinds; ++i) NL_CK(cudaEventCreate(&ev[i]));
  for (int i = 0; i < kNlKinds; ++i) ms[i] = 0.f;
  int rc = SHF_OK;
  for (int it = 0; it < n && rc == SHF_OK; ++it) {
    cudaError_t e = enqueue_nl_iteration(st, ev);
    if (e == cudaSuccess) e = cudaEventSynchronize(ev[kNlKinds]);
    for (int i = 0; i < kNlKinds && e == cudaSuccess; ++i) {
      float t = 0.f;
      e = cudaEventElapsedTime(&t, ev[i], ev[i + 1]);
      ms[i] += t / n;
    }
    if (e != cudaSuccess) rc = nl_fail(SHF_ERR_CUDA, std::string("nl_admm_kernel_times: ") + cudaGetErrorString(e));
  }
  for (int i = 0; i <= kNlKinds; ++i) cudaEventDestroy(ev[i]);
  if (rc == SHF_OK) st->iter += n;
  if (nk) *nk = kNlKinds;
  return rc;
}

const char* nl_admm_kernel_name(int i) { return (i >= 0 && i < kNlKinds) ? kNlNames[i] : ""; }

int nl_admm_get(nl_state* st, int what, void* dst, int on_host) {
  if (!st || !dst) return nl_fail(SHF_ERR_ARG, "nl_admm_get: NULL argument");
  const size_t P = st->P(), K = st->K, m = st->m;
  const cudaMemcpyKind kind = on_host ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
  switch (what) {
    case SEG_U: return nl_copy(st, dst, st->u, sizeof(float) * P * K, kind, on_host);
    case SEG_W: return nl_copy(st, dst, st->w, sizeof(float) * P * K, kind, on_host);
    case SEG_BW: return nl_copy(st, dst, st->bw, sizeof(float) * P * K, kind, on_host);
    case SEG_S: return nl_copy(st, dst, st->s, sizeof(float) * P * K, kind, on_host);
    case SEG_BV:
    case SEG_V: {  // b_v, or v = d + b_v, label-major
      const size_t n = m * P * K;
      float* tgt = static_cast<float*>(dst);
      if (on_host) NL_CK(cudaMallocAsync(reinterpret_cast<void**>(&tgt), sizeof(float) * n, st->stream));
      k_nl_unpack<<<grid_for(m * P * st->Q), kThreads, 0, st->stream>>>(
          what == SEG_V ? st->d : st->bv, what == SEG_V ? st->bv : nullptr, tgt, 1.f, st->K, st->Q, m * P);
      cudaError_t e = cudaGetLastError();
      if (on_host) {
        if (e == cudaSuccess) e = cudaMemcpyAsync(dst, tgt, sizeof(float) * n, cudaMemcpyDeviceToHost, st->stream);
        cudaError_t e2 = cudaFreeAsync(tgt, st->stream);
        if (e == cudaSuccess) e = e2;
        if (e == cudaSuccess) e = cudaStreamSynchronize(st->stream);
      }
      NL_CK(e);
      return SHF_OK;
    }
    case SEG_LABELS:
    case SEG_GAP: {
      NL_CK(shf::launch_labels(st->w, st->K, static_cast<int>(P), st->labels, st->gap, st->stream));
      return nl_copy(st, dst, what == SEG_LABELS ? static_cast<void*>(st->labels) : static_cast<void*>(st->gap),
                     sizeof(float) * P, kind, on_host);
    }
    case SEG_ENERGY: {
      k_nl_energy<<<kRedBlocks, kThreads, 0, st->stream>>>(st->w, st->s, st->nbr, st->deg, st->K, st->m, P,
                                                           st->red + 2);
      NL_CK(cudaGetLastError());
      k_nl_energy_final<<<1, 32, 0, st->stream>>>(st->red + 2, kRedBlocks, st->red);
      NL_CK(cudaGetLastError());
      double hst[2];
      NL_CK(cudaMemcpyAsync(hst, st->red, sizeof(hst), cudaMemcpyDeviceToHost, st->stream));
      NL_CK(cudaStreamSynchronize(st->stream));
      const double energy = hst[0] + static_cast<double>(st->lambda) * hst[1];
      if (on_host) {
        *static_cast<double*>(dst) = energy;
        return SHF_OK;
      }
      return nl_copy(st, dst, &energy, sizeof(double), cudaMemcpyHostToDevice, true);
    }
    case SEG_ITER: {
      if (!on_host) return nl_fail(SHF_ERR_ARG, "SEG_ITER is read into host memory");
      NL_CK(cudaStreamSynchronize(st->stream));
      *static_cast<int*>(dst) = st->iter;
      return SHF_OK;
    }
    default: return nl_fail(SHF_ERR_ARG, "nl_admm_get: unknown selector");
  }
}

int nl_admm_read(nl_state* st, int what, void* dst, void* earlier) {
  if (!st || !dst) return nl_fail(SHF_ERR_ARG, "nl_admm_read: NULL argument");
  NL_CK(shf::order_after(st->stream, static_cast<cudaStream_t>(earlier)));
  const int rc = nl_admm_get(st, what, dst, 0);
  return rc ? rc : nl_admm_sync(st);
}

int nl_admm_set(nl_state* st, int what, const void* src, int on_host) {
  if (!st || !src) return nl_fail(SHF_ERR_ARG, "nl_admm_set: NULL argument");
  const size_t P = st->P(), K = st->K, m = st->m;
  const cudaMemcpyKind kind = on_host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
  int rc = SHF_OK;
  switch (what) {
    case SEG_W: rc = nl_copy(st, st->w, src, sizeof(float) * P * K, kind, false); break;
    case SEG_BW: rc = nl_copy(st, st->bw, src, sizeof(float) * P * K, kind, false); break;
    case SEG_U: rc = nl_copy(st, st->u, src, sizeof(float) * P * K, kind, false); break;
    case SEG_BV:
    case SEG_V: {  // b_v, or d = v - b_v with the current b_v
      const size_t n = m * P * K;
      const float* from = static_cast<const float*>(src);
      float* tmp = nullptr;
      if (on_host) {
        NL_CK(cudaMallocAsync(reinterpret_cast<void**>(&tmp), sizeof(float) * n, st->stream));
        from = tmp;
      }
      cudaError_t e = on_host ? cudaMemcpyAsync(tmp, src, sizeof(float) * n, cudaMemcpyHostToDevice, st->stream) : cudaSuccess;
      if (e == cudaSuccess) {
        k_nl_pack<<<grid_for(m * P * st->Q), kThreads, 0, st->stream>>>(
            from, what == SEG_V ? st->bv : nullptr, what == SEG_V ? st->d : st->bv, -1.f, st->K, st->Q, m * P);
        e = cudaGetLastError();
      }
      if (tmp) {
        const cudaError_t e2 = cudaFreeAsync(tmp, st->stream);
        if (e == cudaSuccess) e = e2;
      }
      NL_CK(e);
      break;
    }
    default: return nl_fail(SHF_ERR_ARG, "nl_admm_set: accepts SEG_W, SEG_BW, SEG_U, SEG_BV and SEG_V");
  }
  if (rc) return rc;
  NL_CK(rebuild_rhs(st));
  NL_CK(cudaStreamSynchronize(st->stream));
  return SHF_OK;
}

int nl_admm_sync(nl_state* st) {
  if (!st) return nl_fail(SHF_ERR_ARG, "nl_admm_sync: NULL state");
  NL_CK(cudaStreamSynchronize(st->stream));
  int gave_up = 0;
  NL_CK(cudaMemcpy(&gave_up, st->cerr, sizeof(int), cudaMemcpyDeviceToHost));
  if (gave_up) {
    NL_CK(cudaMemset(st->cerr, 0, sizeof(int)));
    return nl_fail(SHF_ERR_TIMEOUT, "nl_admm_sync: a grid barrier of the Chebyshev solve gave up");
  }
  return SHF_OK;
}

int nl_admm_barrier_selftest(nl_state* st) {
  if (!st) return nl_fail(SHF_ERR_ARG, "nl_admm_barrier_selftest: NULL state");
  NL_CK(cudaStreamSynchronize(st->stream));
  NL_CK(cudaMemsetAsync(st->cbar, 0, sizeof(unsigned), st->stream));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2);
  cfg.blockDim = dim3(32);
  cfg.stream = st->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  NL_CK(cudaLaunchKernelEx(&cfg, k_barrier_unreachable, st->cbar, st->cerr));
  return nl_admm_sync(st);
}

int nl_admm_destroy(nl_state* st) {
  free_nl(st);
  return SHF_OK;
}

}  // extern "C"
